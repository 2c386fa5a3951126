// The whole CUDA-core step of a small model in one cooperative launch.
//
// A model of a few million parameters is bound by latency: a layer's seven kernels run 2..14 us each, a
// third of that launch, ramp and drain, and the host needs 4 us for every launch.  Here the phases of
// all layers, the LM head, the signals, the cross log-probs and the boundary rule run in one kernel
// of one CTA per SM, with a counting grid barrier between phases.  Two-layer fp32 model (d 256, 96 rows,
// vocab 4096): 22 launches and 157 us per step -> 3 launches and 124 us; a generation step 183 -> 125 us.
//
//   per layer   norm1 + QKV + rotation + cache append | attention | O projection + residual |
//               norm2 + gate / up + SwiGLU | down projection + residual
//   at the end  final norm + LM head | signals | cross log-probs and boundary
//
// A CTA is two groups of 256 threads that work through the tiles (attention units, positions) of a
// phase on their own; a group is what a CTA of the one-launch-per-op kernels is.  The norms have no
// phase: a GEMM tile norms its 16 rows while its weights are on their way, which start before the
// barrier (they depend on nothing).  Data of other CTAs is read past L1 (ld.cg, cp.async.cg).
#include <cuda_runtime.h>

#include "decisions.cuh"
#include "simt_dev.cuh"
#include "simt_step.h"

namespace dc {

namespace {

constexpr int kGroups = 2, kFuseThreads = 256 * kGroups;
constexpr int kKC = 128, kStages = 3;          // k-chunk of the GEMM tiles (16 k per warp), ring stages
constexpr int kCsPitch = 33;
constexpr size_t kGroupSmemMax = 112 * 1024;   // shared memory of a group
constexpr int kMaxNormD = 1024;                // a warp holds a row in registers while it norms it

// How long a thread waits at the grid barrier before it gives up (as in the tensor-core kernels).
__device__ unsigned long long g_simt_wait_ns = 2000000000ull;

struct Group { int id, t, warp, lane, vid, nv; unsigned char* smem; };
__device__ __forceinline__ void gsync(const Group& g) { asm volatile("bar.sync %0, 256;" ::"r"(g.id + 1) : "memory"); }

template <typename T> __device__ __forceinline__ void ldcg4(const T* src, float (&v)[4]);
template <> __device__ __forceinline__ void ldcg4<float>(const float* src, float (&v)[4]) {
  const float4 t = __ldcg(reinterpret_cast<const float4*>(src));
  v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
template <> __device__ __forceinline__ void ldcg4<__nv_bfloat16>(const __nv_bfloat16* src, float (&v)[4]) {
  const uint2 t = __ldcg(reinterpret_cast<const uint2*>(src));
  const __nv_bfloat162 a = *reinterpret_cast<const __nv_bfloat162*>(&t.x);
  const __nv_bfloat162 b = *reinterpret_cast<const __nv_bfloat162*>(&t.y);
  v[0] = __low2float(a); v[1] = __high2float(a); v[2] = __low2float(b); v[3] = __high2float(b);
}

// One GEMM of the step: acc[m, n] = sum_k A[m, k] W[n, k].
template <typename T>
struct FuseGemm {
  const T* A;              // SRC_GLOBAL: [M, K]
  const T *w0, *w1, *w2;
  const T* gain;           // SRC_NORM / SRC_LM: gain of the norm that makes A
  int M, N, K, ldc;
  float* C;
  T* act;
};
enum { SRC_GLOBAL = 0, SRC_NORM = 1, SRC_LM = 2 };

// dst_i = T(rmsnorm(row) * gain) by one warp, into up to three places (null: skipped); columns d ..
// pad_to of s0 are zeroed
template <typename T>
__device__ __forceinline__ void norm_row(const float* row, const T* gain, float eps, int d, T* s0, int pad_to, T* g0, T* g1,
                                         int lane) {
  float4 v[kMaxNormD / 128];
  float ss = 0.f;
#pragma unroll
  for (int i = 0; i < kMaxNormD / 128; ++i) {
    const int e = lane * 4 + 128 * i;
    if (e < d) {
      v[i] = __ldcg(reinterpret_cast<const float4*>(row + e));
      ss += v[i].x * v[i].x + v[i].y * v[i].y + v[i].z * v[i].z + v[i].w * v[i].w;
    }
  }
  ss = warp_sum(ss);
  const float inv = rsqrtf(ss / (float)d + eps);
#pragma unroll
  for (int i = 0; i < kMaxNormD / 128; ++i) {
    const int e = lane * 4 + 128 * i;
    float o[4] = {0.f, 0.f, 0.f, 0.f};
    if (e < d) {
      float gv[4];
      load4<T>(gain + e, gv);
      o[0] = v[i].x * inv * gv[0]; o[1] = v[i].y * inv * gv[1]; o[2] = v[i].z * inv * gv[2]; o[3] = v[i].w * inv * gv[3];
      if (g0) store4<T>(g0 + e, o);
      if (g1) store4<T>(g1 + e, o);
    }
    if (s0 && e < pad_to) store4<T>(s0 + e, o);
  }
}
template <typename T>
__device__ __forceinline__ void copy_row(const T* src, int d, T* s0, int pad_to, T* g0, int lane) {   // src null: zeros
  for (int e = lane * 4; e < pad_to; e += 128) {
    float o[4] = {0.f, 0.f, 0.f, 0.f};
    if (src != nullptr && e < d) ldcg4<T>(src + e, o);
    store4<T>(s0 + e, o);
    if (g0 && e < d) store4<T>(g0 + e, o);
  }
}

// LM-head input row lrow (see k_lm_rows) into s0; `own`: also into h (and the curr rows into h_out)
template <typename T>
__device__ __forceinline__ void lm_row_to(const SimtStep<T>& p, int lrow, T* s0, int pad_to, bool own, int lane) {
  const SeqMeta& m = p.ml;
  const int grp = lrow / (m.nv * m.G), in = lrow % (m.nv * m.G);
  const int v = in / m.G, pos = grp * m.G + in % m.G;
  const int b = pos / m.W_cap, k = pos % m.W_cap;
  T* hr = own ? p.h + (size_t)lrow * p.d : nullptr;
  if (lrow >= m.nv * m.npos_pad || b >= m.batch || k >= m.win_len[b]) {
    copy_row<T>(nullptr, p.d, s0, pad_to, lrow < m.nv * m.npos_pad ? hr : nullptr, lane);
    return;
  }
  T* ho = (own && v == 0 && p.io.h_out != nullptr) ? p.io.h_out + ((size_t)b * p.max_window + k) * p.d : nullptr;
  const T* src = p.io.h_in != nullptr ? p.io.h_in + (((size_t)b * 2 + v) * p.max_window + k) * p.d
               : (v >= p.m.nv && k < p.io.prev.n[b]) ? p.io.h_prev_in + ((size_t)b * p.max_window + k) * p.d : nullptr;
  if (src != nullptr) {
    copy_row<T>(src, p.d, s0, pad_to, hr, lane);
    if (ho == nullptr || p.io.h_in == nullptr) return;
    s0 = nullptr; hr = nullptr;
  }
  norm_row<T>(p.x + (size_t)act_row(p.m, v < p.m.nv ? v : 0, b, p.m.last_len[b] + k) * p.d, p.final_norm, p.eps, p.d, s0,
              pad_to, hr, ho, lane);
}

// what simt_store_qkv needs
template <typename T>
struct QkvView {
  const SeqMeta& m;
  int nq, nkv, hd, max_ctx;
  const float* cos_sin;
  const T *bq, *bk, *bv;
  T *q, *k, *v, *k_cache, *v_cache;
};

// All tiles (16 rows x 32 columns, as in k_gemm_simt) of one GEMM; `wait` is the barrier in front of the
// phase: every thread of the CTA calls it once.  Returns false if it gave up.
template <typename T, int EPI, int SRC, typename Wait>
__device__ bool gemm_phase(const SimtStep<T>& p, const FuseGemm<T>& g, const QkvView<T>* qv, const Group& gr, Wait&& wait) {
  constexpr int PIECE = GemmIo<T>::kPiece, PITCH = kKC + GemmIo<T>::kPad, PPR = kKC / PIECE;   // pieces per row of a chunk
  constexpr int WR = 32 * PPR / 256, AR = 16 * PPR / 256;      // rows of W / A that a thread copies a piece of
  constexpr int RSTEP = 256 / PPR;
  const int chunks = (g.K + kKC - 1) / kKC, apitch = SRC == SRC_GLOBAL ? PITCH : chunks * kKC + GemmIo<T>::kPad;
  T* ring_w = reinterpret_cast<T*>(gr.smem);                    // [stages][32][PITCH]
  T* as = ring_w + kStages * 32 * PITCH;                        // [stages][16][PITCH], or the 16 whole rows
  float* cs = reinterpret_cast<float*>(as + (SRC == SRC_GLOBAL ? kStages * 16 * PITCH : 16 * apitch));   // [8][16][33]
  const int units = EPI == EPI_QKV ? (p.nq + 2 * p.nkv) * (p.hd / 32) : EPI == EPI_SWIGLU ? (g.N + 15) / 16 : (g.N + 31) / 32;
  const int MT = (g.M + 15) / 16, tiles = MT * units;
  const int r_t = gr.t / PPR, k_t = (gr.t % PPR) * PIECE;
  const int ty = gr.lane >> 3, tx = gr.lane & 7;
  bool waited = false;
  for (int tile = gr.vid; tile < tiles || !waited; tile += gr.nv) {
    const bool has = tile < tiles;
    const int u = tile / MT, m0 = (tile - u * MT) * 16;
    const T* wsrc[WR];
    auto load_w = [&](int c) {
      T* dst = ring_w + (size_t)(c % kStages) * 32 * PITCH;
      const int k0 = c * kKC + k_t, bytes = max(0, min(16, (g.K - k0) * (int)sizeof(T)));
#pragma unroll
      for (int i = 0; i < WR; ++i)
        cp_async16(dst + (r_t + i * RSTEP) * PITCH + k_t, wsrc[i] != nullptr && bytes ? wsrc[i] + k0 : g.w0,
                   wsrc[i] != nullptr ? bytes : 0);
    };
    auto load_a = [&](int c) {
      T* dst = as + (size_t)(c % kStages) * 16 * PITCH;
      const int k0 = c * kKC + k_t, bytes = max(0, min(16, (g.K - k0) * (int)sizeof(T)));
#pragma unroll
      for (int i = 0; i < (AR > 0 ? AR : 1); ++i) {
        const int r = r_t + i * RSTEP;
        const bool in = m0 + r < g.M && bytes > 0;
        cp_async16(dst + r * PITCH + k_t, in ? g.A + (size_t)(m0 + r) * g.K + k0 : g.A, in ? bytes : 0);
      }
    };
    if (has) {
#pragma unroll
      for (int i = 0; i < WR; ++i) {
        const int jj = r_t + i * RSTEP;
        const T* src = nullptr;
        if (EPI == EPI_QKV) {
          const int half = p.hd >> 1, per_head = p.hd >> 5, head = u / per_head;
          const int e = (u - head * per_head) * 16 + (jj & 15) + (jj >> 4) * half;
          if (head < p.nq) src = g.w0 + (size_t)(head * p.hd + e) * g.K;
          else if (head < p.nq + p.nkv) src = g.w1 + (size_t)((head - p.nq) * p.hd + e) * g.K;
          else src = g.w2 + (size_t)((head - p.nq - p.nkv) * p.hd + e) * g.K;
        } else if (EPI == EPI_SWIGLU) {
          const int f = u * 16 + (jj & 15);
          if (f < g.N) src = (jj < 16 ? g.w0 : g.w1) + (size_t)f * g.K;
        } else {
          const int n = u * 32 + jj;
          if (n < g.N) src = g.w0 + (size_t)n * g.K;
        }
        wsrc[i] = src;
      }
      for (int c = 0; c < kStages - 1 && c < chunks; ++c) load_w(c);
    }
    if (!waited) {
      if (!wait()) return false;
      waited = true;
    }
    if (!has) break;
    float old[2];   // residual values that the epilogue adds to
    if (EPI == EPI_ADD_F32) {
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int pos = gr.t + 256 * i, r = pos >> 5, n = u * 32 + (pos & 31);
        old[i] = (m0 + r < g.M && n < g.N) ? __ldcg(g.C + (size_t)(m0 + r) * g.ldc + n) : 0.f;
      }
    }
    if (SRC == SRC_GLOBAL) {   // group c: W chunk c (all W loads so far with the first) and A chunk c
      for (int c = 0; c < kStages - 1; ++c) {
        if (c < chunks) load_a(c);
        asm volatile("cp.async.commit_group;" ::: "memory");
      }
    } else {
      for (int c = 0; c < kStages - 1; ++c) asm volatile("cp.async.commit_group;" ::: "memory");
#pragma unroll 1
      for (int i = 0; i < 2; ++i) {
        const int r = gr.warp * 2 + i, row = m0 + r;
        T* dst = as + (size_t)r * apitch;
        if (SRC == SRC_LM) lm_row_to<T>(p, row, dst, chunks * kKC, u == 0, gr.lane);
        else if (row < g.M) norm_row<T>(p.x + (size_t)row * p.d, g.gain, p.eps, p.d, dst, chunks * kKC, (T*)nullptr, (T*)nullptr, gr.lane);
        else copy_row<T>(nullptr, p.d, dst, chunks * kKC, nullptr, gr.lane);
      }
    }
    f2 acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
    for (int c = 0; c < chunks; ++c) {
      asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
      gsync(gr);               // chunk c has landed for every thread; the stage of chunk c - 1 is free
      if (c + kStages - 1 < chunks) {
        load_w(c + kStages - 1);
        if (SRC == SRC_GLOBAL) load_a(c + kStages - 1);
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
      const T* wp = ring_w + (size_t)(c % kStages) * 32 * PITCH + tx * PITCH + gr.warp * (kKC / 8);
      const T* ap = (SRC == SRC_GLOBAL ? as + (size_t)(c % kStages) * 16 * PITCH : as + c * kKC) + ty * 4 * apitch + gr.warp * (kKC / 8);
#pragma unroll
      for (int k = 0; k < kKC / 8; k += 4) {
        f2 av[4][2], wv[4][2];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          float v[4];
          load4<T>(ap + i * apitch + k, v);
          av[i][0] = pack2(v[0], v[1]); av[i][1] = pack2(v[2], v[3]);
          load4<T>(wp + i * 8 * PITCH + k, v);
          wv[i][0] = pack2(v[0], v[1]); wv[i][1] = pack2(v[2], v[3]);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            fma2(acc[i][j], av[i][0], wv[j][0]);
            fma2(acc[i][j], av[i][1], wv[j][1]);
          }
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) cs[(gr.warp * 16 + ty * 4 + i) * kCsPitch + tx + 8 * j] = sum2(acc[i][j]);
    gsync(gr);                 // the sums are there, and the ring and the rows have been read
    auto value = [&](int r, int c) {
      float v = cs[r * kCsPitch + c];
#pragma unroll
      for (int w = 1; w < 8; ++w) v += cs[(w * 16 + r) * kCsPitch + c];
      return v;
    };
    if (EPI == EPI_STORE_F32 || EPI == EPI_ADD_F32) {
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int pos = gr.t + 256 * i, r = pos >> 5, c = pos & 31, n = u * 32 + c;
        if (m0 + r < g.M && n < g.N) g.C[(size_t)(m0 + r) * g.ldc + n] = EPI == EPI_ADD_F32 ? old[i] + value(r, c) : value(r, c);
      }
    } else {
      const int r = gr.t >> 4, i = gr.t & 15, m = m0 + r;
      if (m < g.M) {
        const float y1 = value(r, i), y2 = value(r, 16 + i);
        if (EPI == EPI_SWIGLU) {
          const int f = u * 16 + i;
          if (f < g.N) g.act[(size_t)m * g.N + f] = from_f<T>(y1 / (1.f + expf(-y1)) * y2);
        } else {
          const int per_head = p.hd >> 5, head = u / per_head;
          simt_store_qkv<T>(*qv, m, head, (u - head * per_head) * 16 + i, y1, y2);
        }
      }
    }
  }
  return true;
}

// Bidirectional attention: a unit is 8 query rows of one head and variant, a row per warp.  Tiles of
// p.kt keys arrive in two buffers as they lie in memory (cached V transposed, active V row-major).
template <typename T, typename Wait>
__device__ bool attn_phase(const SimtStep<T>& p, int layer, const Group& gr, Wait&& wait) {
  constexpr int PIECE = GemmIo<T>::kPiece;
  const SeqMeta& m = p.m;
  const int hd = p.hd, kt = p.kt, kp = hd + PIECE, vp = kt + PIECE;
  const int vbuf = max(kt * kp, hd * vp);
  T* kb = reinterpret_cast<T*>(gr.smem);             // [2][kt][kp]
  T* vb = kb + 2 * kt * kp;                          // [2][vbuf]
  float* qs = reinterpret_cast<float*>(vb + 2 * vbuf) + gr.warp * (hd + kt);   // this warp's query row, then its probabilities
  float* ps = qs + hd;
  const int nrt = (m.R_cap + 7) / 8, units = nrt * p.nq * m.nv * m.batch, ld = p.nkv * hd;
  const float scale = rsqrtf((float)hd);
  bool waited = false;
  for (int unit = gr.vid; unit < units || !waited; unit += gr.nv) {
    const bool has = unit < units;
    const int vbi = unit / (nrt * p.nq), rem = unit - vbi * nrt * p.nq, h = rem / nrt, r0 = (rem - h * nrt) * 8;
    const int b = has ? vbi % m.batch : 0, vv = vbi / m.batch;
    const int P = m.ctx_len[b], R = m.last_len[b] + m.win_len[b], kvh = h / (p.nq / p.nkv);
    const int row0 = act_row(m, vv, b, 0);
    const int tc = (P + kt - 1) / kt, nt = (has && r0 < R) ? tc + (R + kt - 1) / kt : 0;
    const size_t kv = (size_t)layer * p.cache_layer + ((size_t)b * p.nkv + kvh) * (size_t)p.max_ctx * hd;
    auto load = [&](int t) {
      if (t < nt) {
        const bool ctx = t < tc;
        const int j0 = (ctx ? t : t - tc) * kt, n = min(kt, (ctx ? P : R) - j0), hq = hd / PIECE;
        T* kd = kb + (size_t)(t & 1) * kt * kp;
        T* vd = vb + (size_t)(t & 1) * vbuf;
        for (int i = gr.t; i < kt * hq; i += 256) {
          const int j = i / hq, e = (i - j * hq) * PIECE;
          const T* src = ctx ? p.k_cache + kv + (size_t)(j0 + j) * hd + e : p.k + (size_t)(row0 + j0 + j) * ld + kvh * hd + e;
          cp_async16(kd + j * kp + e, j < n ? src : p.k, j < n ? 16 : 0);
          if (!ctx) {
            const T* vs = p.v + (size_t)(row0 + j0 + j) * ld + kvh * hd + e;
            cp_async16(vd + j * kp + e, j < n ? vs : p.v, j < n ? 16 : 0);
          }
        }
        if (ctx) {   // keys are contiguous; what the cache holds beyond ctx_len is not read
          const int kq = kt / PIECE;
          for (int i = gr.t; i < hd * kq; i += 256) {
            const int e = i / kq, j = (i - e * kq) * PIECE, bytes = max(0, min(16, (n - j) * (int)sizeof(T)));
            cp_async16(vd + e * vp + j, bytes ? p.v_cache + kv + (size_t)e * p.max_ctx + j0 + j : p.v, bytes);
          }
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    const bool early = !waited && nt > 0 && tc > 0;   // the first cached tile depends on nothing
    if (early) load(0);
    if (!waited) {
      if (!wait()) return false;
      waited = true;
    }
    if (!has) break;
    if (nt == 0) continue;
    if (!early) load(0);
    const int row = r0 + gr.warp;
    const bool live = row < R;
    if (live)
      for (int e = gr.lane * 4; e < hd; e += 128) {
        float v[4];
        ldcg4<T>(p.q + (size_t)(row0 + row) * p.nq * hd + (size_t)h * hd + e, v);
        *reinterpret_cast<float4*>(qs + e) = make_float4(v[0], v[1], v[2], v[3]);
      }
    float mx = -INFINITY, sum = 0.f, o[4] = {0.f, 0.f, 0.f, 0.f};
    for (int t = 0; t < nt; ++t) {
      load(t + 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
      gsync(gr);
      if (live) {
        const bool ctx = t < tc;
        const int n = min(kt, ctx ? P - t * kt : R - (t - tc) * kt);
        const T* kd = kb + (size_t)(t & 1) * kt * kp;
        const T* vd = vb + (size_t)(t & 1) * vbuf;
        float tm = -INFINITY;
        for (int j = gr.lane; j < kt; j += 32) {   // one key per lane and step
          float s = -INFINITY;
          if (j < n) {
            float a0 = 0.f, a1 = 0.f;
            const T* kr = kd + j * kp;
#pragma unroll 4
            for (int e = 0; e < hd; e += 4) {
              float x[4];
              load4<T>(kr + e, x);
              const float4 qv = *reinterpret_cast<const float4*>(qs + e);
              a0 = fmaf(qv.x, x[0], a0); a1 = fmaf(qv.y, x[1], a1); a0 = fmaf(qv.z, x[2], a0); a1 = fmaf(qv.w, x[3], a1);
            }
            s = (a0 + a1) * scale;
          }
          ps[j] = s;
          tm = fmaxf(tm, s);
        }
        const float nm = fmaxf(mx, warp_max(tm)), corr = expf(mx - nm);   // 0 on the first tile
        float ts = 0.f;
        for (int j = gr.lane; j < kt; j += 32) {
          const float e = expf(ps[j] - nm);
          ps[j] = e;
          ts += e;
        }
        sum = sum * corr + warp_sum(ts);
        mx = nm;
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int e = gr.lane + 32 * i;
          if (e < hd) {
            float x0 = 0.f, x1 = 0.f;
            if (ctx) {
              const T* vr = vd + e * vp;
#pragma unroll 4
              for (int j = 0; j < kt; j += 4) {
                float w[4];
                load4<T>(vr + j, w);
                const float4 pv = *reinterpret_cast<const float4*>(ps + j);
                x0 = fmaf(pv.x, w[0], x0); x1 = fmaf(pv.y, w[1], x1); x0 = fmaf(pv.z, w[2], x0); x1 = fmaf(pv.w, w[3], x1);
              }
            } else {
#pragma unroll 8
              for (int j = 0; j < kt; j += 2) {
                x0 = fmaf(ps[j], to_f<T>(vd[j * kp + e]), x0);
                x1 = fmaf(ps[j + 1], to_f<T>(vd[(j + 1) * kp + e]), x1);
              }
            }
            o[i] = o[i] * corr + (x0 + x1);
          }
        }
      }
      gsync(gr);
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    if (live) {
      const float inv = 1.f / sum;
      T* dst = p.o + (size_t)(row0 + row) * p.nq * hd + (size_t)h * hd;
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (gr.lane + 32 * i < hd) dst[gr.lane + 32 * i] = from_f<T>(o[i] * inv);
    }
  }
  return true;
}

// Cross log-probs (Eq. 6 halves): xlogp[b,i,j] = h_i . W_lm[yhat_j] - lse_i.  A unit is a column j and 16
// rows; every warp keeps its part of W_lm[yhat_j] in registers.
template <typename T>
__device__ __forceinline__ void xlogp_phase(const SimtStep<T>& p, const Group& gr) {
  const SeqMeta& m = p.ml;
  const int it = (m.W_cap + 15) / 16, units = m.batch * m.W_cap * it;
  for (int unit = gr.vid; unit < units; unit += gr.nv) {
    const int bj = unit / it, b = bj / m.W_cap, j = bj - b * m.W_cap, W = m.win_len[b];
    if (j >= W) continue;
    const int tok = __ldcg(p.sig.ws_pred + b * m.W_cap + j);
    const bool ok = tok >= 0 && tok < p.V;   // never index the vocabulary matrix with an id outside it
    float w[kMaxNormD / 128][4];
#pragma unroll
    for (int i = 0; i < kMaxNormD / 128; ++i)
      if (ok && gr.lane * 4 + 128 * i < p.d) load4<T>(p.lm_head + (size_t)tok * p.d + gr.lane * 4 + 128 * i, w[i]);
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int i0 = (unit - bj * it) * 16 + gr.warp * 2 + r;
      if (i0 >= W) continue;
      const T* hr = p.h + (size_t)lm_row(m, 0, b * m.W_cap + i0) * p.d;
      float acc = 0.f;
#pragma unroll
      for (int i = 0; i < kMaxNormD / 128; ++i)
        if (gr.lane * 4 + 128 * i < p.d) {
          float hv[4];
          ldcg4<T>(hr + gr.lane * 4 + 128 * i, hv);
#pragma unroll
          for (int c = 0; c < 4; ++c) acc = fmaf(hv[c], ok ? w[i][c] : 0.f, acc);
        }
      acc = warp_sum(acc);
      if (gr.lane == 0)
        p.xlogp[((size_t)b * p.max_window + i0) * p.max_window + j] = ok ? acc - __ldcg(p.sig.ws_lse + b * m.W_cap + i0) : -INFINITY;
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(kFuseThreads, 1) k_simt_step(const __grid_constant__ SimtStep<T> p) {
  extern __shared__ __align__(16) unsigned char fuse_smem[];
  __shared__ int go;
  __shared__ SignalsShared<256> sig_sh[kGroups];
  __shared__ float bnd[2][33 * (DC_MAX_WINDOW / 32)];
  Group gr;
  gr.id = threadIdx.x >> 8; gr.t = threadIdx.x & 255; gr.warp = gr.t >> 5; gr.lane = gr.t & 31;
  gr.vid = gr.id * gridDim.x + blockIdx.x;   // the first tiles of a phase go to different SMs
  gr.nv = kGroups * gridDim.x;
  gr.smem = fuse_smem + (size_t)gr.id * p.group_smem;

  // Grid barrier: a CTA counts itself in when all of its threads are through a phase and goes on (its
  // next weights do not depend on the others) until it needs what they wrote.
  unsigned int target = 0;
  auto arrive = [&]() {
    __syncthreads();
    target += gridDim.x;
    if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p.bar) : "memory");
  };
  auto wait = [&]() -> bool {
    if (target == 0u) return true;
    if (threadIdx.x == 0) {
      unsigned long long t0 = 0ull, now;
      unsigned int v, polls = 0;
      int ok = 1;
      while (true) {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p.bar) : "memory");
        if (v >= target) break;
        if ((++polls & 0x3f) == 0) {
          asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
          if (t0 == 0ull) t0 = now;
          asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p.bar + 1) : "memory");
          if (v != 0u || now - t0 > g_simt_wait_ns) {
            ok = 0;
            atomicExch(p.bar + 1, 1u);   // the CTAs still waiting give up too
            for (int b = 0; b < p.m.batch; ++b) atomicExch(p.sig.status + b, (int)DC_ERR_TIMEOUT);
            break;
          }
        }
      }
      go = ok;
    }
    __syncthreads();
    return go != 0;
  };

  const int M = p.m.nv * p.m.batch * p.m.R_cap;
  for (int l = 0; l < p.n_layers; ++l) {
    const SimtLayer<T> L = p.layers[l];
    const size_t cache = (size_t)l * p.cache_layer;
    const QkvView<T> qv{p.m, p.nq, p.nkv, p.hd, p.max_ctx, p.cos_sin, L.bq, L.bk, L.bv, p.q, p.k, p.v,
                        p.export_kv ? p.k_cache + cache : nullptr, p.export_kv ? p.v_cache + cache : nullptr};
    if (!gemm_phase<T, EPI_QKV, SRC_NORM>(p, FuseGemm<T>{nullptr, L.wq, L.wk, L.wv, L.n1, M, 0, p.d, 0, nullptr, nullptr}, &qv, gr, wait)) return;
    if (p.kv_only && l + 1 == p.n_layers) return;
    arrive();
    if (!attn_phase<T>(p, l, gr, wait)) return;
    arrive();
    if (!gemm_phase<T, EPI_ADD_F32, SRC_GLOBAL>(p, FuseGemm<T>{p.o, L.wo, nullptr, nullptr, nullptr, M, p.d, p.nq * p.hd, p.d, p.x, nullptr}, nullptr, gr, wait)) return;
    arrive();
    if (!gemm_phase<T, EPI_SWIGLU, SRC_NORM>(p, FuseGemm<T>{nullptr, L.wg, L.wu, nullptr, L.n2, M, p.F, p.d, 0, nullptr, p.act}, nullptr, gr, wait)) return;
    arrive();
    if (!gemm_phase<T, EPI_ADD_F32, SRC_GLOBAL>(p, FuseGemm<T>{p.act, L.wd, nullptr, nullptr, nullptr, M, p.d, p.F, p.d, p.x, nullptr}, nullptr, gr, wait)) return;
    arrive();
  }
  if (!gemm_phase<T, EPI_STORE_F32, SRC_LM>(p, FuseGemm<T>{nullptr, p.lm_head, nullptr, nullptr, p.final_norm, p.ml.nv * p.ml.npos_pad, p.V, p.d, p.V, p.logits, nullptr}, nullptr, gr, wait)) return;
  arrive();
  if (!wait()) return;
  for (int pos = gr.vid; pos < p.ml.batch * p.ml.W_cap; pos += gr.nv) {
    signals_pos<256>(p.sig, p.ml, pos, gr.t, sig_sh[gr.id], [&] { gsync(gr); });
    gsync(gr);
  }
  arrive();
  if (!wait()) return;
  if (p.xlogp != nullptr) xlogp_phase<T>(p, gr);
  if (p.bnd.block_len != nullptr && gr.id == 0 && gr.warp == 0)   // the SMs that get the fewest cross log-prob units
    for (int b = gridDim.x - 1 - blockIdx.x; b < p.ml.batch; b += gridDim.x)
      boundary_seq<DC_MAX_WINDOW / 32>(p.sig.ws_infl, p.sig.ws_ent, b, p.ml, DevLens{}, p.hp, p.bnd, bnd[0], bnd[1]);
}

template <typename T>
size_t group_smem(int d, int hd, int kt) {
  const size_t pitch = kKC + GemmIo<T>::kPad, rows = (size_t)(d + kKC - 1) / kKC * kKC + GemmIo<T>::kPad;
  const size_t a = 16 * (kStages * pitch > rows ? kStages * pitch : rows);
  const size_t gemm = (kStages * 32 * pitch + a) * sizeof(T) + 8 * 16 * kCsPitch * sizeof(float);
  const size_t kp = hd + GemmIo<T>::kPiece, vp = kt + GemmIo<T>::kPiece;
  const size_t vb = kt * kp > hd * vp ? kt * kp : hd * vp;
  const size_t attn = 2 * (kt * kp + vb) * sizeof(T) + 8 * (size_t)(hd + kt) * sizeof(float);
  return ((gemm > attn ? gemm : attn) + 127) / 128 * 128;
}

}  // namespace

template <typename T>
bool simt_step_init(SimtFuse* f, int d, int F, int nq, int nkv, int hd, int vocab, int max_ctx) {
  *f = SimtFuse{};
  constexpr int PIECE = GemmIo<T>::kPiece;
  // rows that copies of 16 bytes can tile, and the shapes the phases are written for
  if (hd % 32 || hd > 128 || d % PIECE || F % PIECE || d > kMaxNormD || max_ctx % PIECE) return true;
  f->kt = 64;
  f->group_smem = (int)group_smem<T>(d, hd, f->kt);
  if ((size_t)f->group_smem > kGroupSmemMax) {
    f->kt = 32;
    f->group_smem = (int)group_smem<T>(d, hd, f->kt);
  }
  if ((size_t)f->group_smem > kGroupSmemMax) return true;
  int dev = 0, coop = 0, sms = 0, per_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (!coop || sms < 1) return true;
  if (cudaFuncSetAttribute(k_simt_step<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kGroups * kGroupSmemMax)) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_simt_step<T>, kFuseThreads, kGroups * f->group_smem) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  if (per_sm >= 1) f->grid = sms;
  return true;
}

template <typename T>
bool simt_step_ok(const SimtFuse& f, const SimtStep<T>& p) {
  if (f.grid == 0) return false;
  // GEMMs that take many rounds of small tiles are better off as kernels of their own, with the larger tile
  const long long M = (long long)p.m.nv * p.m.batch * p.m.R_cap, Mlm = (long long)p.ml.nv * p.ml.npos_pad;
  const long long mt = (M + 15) / 16;
  long long most = mt * ((p.F + 15) / 16);
  const long long qkv = mt * (p.nq + 2 * p.nkv) * (p.hd / 32), lm = p.kv_only ? 0 : (Mlm + 15) / 16 * ((p.V + 31) / 32);
  most = most > qkv ? most : qkv;
  most = most > lm ? most : lm;
  return most <= kFuseMaxTiles;
}

template <typename T>
int launch_simt_step(const SimtFuse& f, SimtStep<T> p, cudaStream_t s) {
  p.kt = f.kt; p.group_smem = f.group_smem;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(f.grid); cfg.blockDim = dim3(kFuseThreads);
  cfg.dynamicSmemBytes = (size_t)kGroups * f.group_smem; cfg.stream = s;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeCooperative;
  attr.val.cooperative = 1;
  cfg.attrs = &attr; cfg.numAttrs = 1;
  return (int)cudaLaunchKernelEx(&cfg, k_simt_step<T>, p);
}

int simt_set_wait_limit_us(long long us, cudaStream_t s) {
  const unsigned long long ns = (unsigned long long)us * 1000ull;
  cudaError_t e = cudaMemcpyToSymbolAsync(g_simt_wait_ns, &ns, sizeof(ns), 0, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  return (int)e;
}

#define DC_INST_STEP(T)                                                              \
  template bool simt_step_init<T>(SimtFuse*, int, int, int, int, int, int, int);    \
  template bool simt_step_ok<T>(const SimtFuse&, const SimtStep<T>&);                \
  template int launch_simt_step<T>(const SimtFuse&, SimtStep<T>, cudaStream_t);
DC_INST_STEP(float)
DC_INST_STEP(__nv_bfloat16)

}  // namespace dc
