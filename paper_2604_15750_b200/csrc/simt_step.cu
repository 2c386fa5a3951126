// The whole CUDA-core step of a small model in one cooperative launch.
//
// A model of a few million parameters is bound by latency: a layer's seven kernels run 2..14 us each, a
// third of that launch, ramp and drain, and the host needs 4 us for every launch.  Here the phases of
// all layers, the LM head, the signals, the cross log-probs and the boundary rule run in one kernel
// of one CTA per SM, with a counting grid barrier between phases.  Two-layer fp32 model (d 256, 96 rows,
// vocab 4096): 22 launches and 157 us per step -> 3 launches and 100 us; a generation step 183 -> 103 us.
// What is left (clocks of a step's 175 k): 12 barriers, 4100 .. 5300 from the arrival to the first use where the weights
// of two chunks are started in between (4490 of it, the poll behind it 700) and 2500 where nothing is; the norm
// of 16 rows 3700; a tile 3200, with its epilogue 4500.  The first context of a process on a
// device loads the kernel when it is made (dc_create 7..16 ms instead of 0.9).
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

#include <atomic>

#include "decisions.cuh"
#include "simt_dev.cuh"
#include "simt_step.h"

namespace dc {

namespace {

constexpr int kGroups = 2, kFuseThreads = 256 * kGroups;
constexpr int kKC = 256, kStages = 3;          // k-chunk of the GEMM tiles (32 k per warp), ring stages
constexpr size_t kGroupSmemMax = 112 * 1024;   // shared memory of a group
constexpr int kMaxNormD = 1024;                // half a warp norms a row (norm_row), 64 elements of it at this width

// How long a thread waits at the grid barrier before it gives up (as in the tensor-core kernels).
__device__ unsigned long long g_simt_wait_ns = 2000000000ull;

struct Group { int id, t, warp, lane, vid, nv; unsigned char* smem; };
__device__ __forceinline__ void gsync(const Group& g) { asm volatile("bar.sync %0, 256;" ::"r"(g.id + 1) : "memory"); }

// x, for the compiler a new value: what is derived from it is worked out again where it stands instead of being held in
// registers over a whole phase.  (The 32 sums of a tile leave none for that: 2 to 4 spilled ones cost 1.5% of a step.)
__device__ __forceinline__ int afresh(int x) { asm volatile("" : "+r"(x)); return x; }

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
  int epi, src;
};
enum { SRC_GLOBAL = 0, SRC_NORM = 1, SRC_LM = 2 };

// dst_i = T(rmsnorm(row) * gain) by half a warp (lane l of 16), into up to three places (null: skipped);
// columns d .. pad_to of s0 are zeroed.  `row` null: nothing but zeros in s0.  (Loops stay rolled all
// over this file: code that runs once or twice per phase costs its instruction fetches, about 14
// clocks an instruction; unrolled it took 4500 clocks for 256 columns.)
template <typename T>
__device__ __forceinline__ void norm_row(const float* row, const T* gain, float eps, int d, T* s0, int pad_to, T* g0, T* g1,
                                         int l) {
  float ss = 0.f;
#pragma unroll 4
  for (int e = l * 4; e < d; e += 64) {
    const float4 v = row != nullptr ? __ldcg(reinterpret_cast<const float4*>(row + e)) : make_float4(0.f, 0.f, 0.f, 0.f);
    ss += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
    if (sizeof(T) == 4 && s0) {   // the gain now: its latency would follow the row's otherwise
      float gv[4];
      load4<T>(gain + e, gv);
      *reinterpret_cast<float4*>(s0 + e) = make_float4(v.x * gv[0], v.y * gv[1], v.z * gv[2], v.w * gv[3]);
    }
  }
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  const float inv = rsqrtf(ss / (float)d + eps);
#pragma unroll 2
  for (int e = l * 4; e < d; e += 64) {
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    float gv[4] = {1.f, 1.f, 1.f, 1.f};
    if (sizeof(T) == 4 && s0) v = *reinterpret_cast<const float4*>(s0 + e);
    else {
      if (row != nullptr) v = __ldcg(reinterpret_cast<const float4*>(row + e));
      load4<T>(gain + e, gv);
    }
    const float o[4] = {v.x * inv * gv[0], v.y * inv * gv[1], v.z * inv * gv[2], v.w * inv * gv[3]};
    if (s0) store4<T>(s0 + e, o);
    if (g0) store4<T>(g0 + e, o);
    if (g1) store4<T>(g1 + e, o);
  }
  const float z[4] = {0.f, 0.f, 0.f, 0.f};
  if (s0)
    for (int e = d + l * 4; e < pad_to; e += 64) store4<T>(s0 + e, z);
}

// LM-head input row lrow (see k_lm_rows), by half a warp.  A copied row goes into s0 here and false is
// returned; otherwise xr (null: zeros) is the row to norm.  g0, g1: where the normed row goes besides -
// with `own` h, and h_out for the curr rows.
template <typename T>
__device__ __forceinline__ bool lm_row(const SimtStep<T>& p, int lrow, T* s0, int pad_to, bool own, int l, const float*& xr,
                                       T*& g0, T*& g1) {
  const SeqMeta& m = p.ml;
  const int grp = lrow / (m.nv * m.G), in = lrow % (m.nv * m.G);
  const int v = in / m.G, pos = grp * m.G + in % m.G;
  const int b = pos / m.W_cap, k = pos % m.W_cap;
  const bool row_ok = lrow < m.nv * m.npos_pad;
  g0 = own && row_ok ? p.h + (size_t)lrow * p.d : nullptr;
  if (!row_ok || b >= m.batch || k >= m.win_len[b]) return true;
  if (own && v == 0 && p.io.h_out != nullptr) g1 = p.io.h_out + ((size_t)b * p.max_window + k) * p.d;
  xr = p.x + (size_t)act_row(p.m, v < p.m.nv ? v : 0, b, p.m.last_len[b] + k) * p.d;
  const T* src = p.io.h_in != nullptr ? p.io.h_in + (((size_t)b * 2 + v) * p.max_window + k) * p.d
                 : (v >= p.m.nv && k < p.io.prev.n[b]) ? p.io.h_prev_in + ((size_t)b * p.max_window + k) * p.d : nullptr;
  if (src == nullptr) return true;
#pragma unroll 4
  for (int e = l * 4; e < p.d; e += 64) {
    float o[4];
    ldcg4<T>(src + e, o);
    store4<T>(s0 + e, o);
    if (g0) store4<T>(g0 + e, o);
  }
  const float z[4] = {0.f, 0.f, 0.f, 0.f};
  for (int e = p.d + l * 4; e < pad_to; e += 64) store4<T>(s0 + e, z);
  g0 = nullptr;
  if (p.io.h_in == nullptr) g1 = nullptr;
  return false;
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

// All tiles (16 rows x 16 columns; for the epilogues that combine two features 8 and their partners) of
// one GEMM; `wait` is the barrier in front of the phase: every thread of the CTA calls it once.  Returns
// false if it gave up.
//
// A group keeps one row tile and walks through column units, so its rows are normed once; the k-chunks
// of all of its units are one stream through the ring, so that a unit's first loads run under the
// unit before.  Epilogue and source of A are run-time values: one piece of code serves all GEMMs of the
// step and stays in the instruction cache (five instances of it: 5000 clocks for the first chunk of a
// phase, 1500 for the fourth).
template <typename T, typename Wait>
__device__ __forceinline__ bool gemm_phase(const SimtStep<T>& p, const FuseGemm<T>& g, const QkvView<T>& qv, const Group& gr, Wait&& wait) {
  constexpr int KC = kKC, ST = kStages, NC = 16;
  constexpr int PIECE = GemmIo<T>::kPiece, PITCH = KC + GemmIo<T>::kPad, PPR = KC / PIECE;  // pieces per row of a chunk
  constexpr int NP = NC * PPR / 256, RS = 256 / PPR;            // pieces of W (and of A) that a thread copies, rows apart
  constexpr int CP = NC + 1;
  const int chunks = (g.K + KC - 1) / KC, epi = g.epi;
  const bool stream_a = g.src == SRC_GLOBAL;
  const int apitch = stream_a ? PITCH : chunks * KC + GemmIo<T>::kPad;
  T* ring_w = reinterpret_cast<T*>(gr.smem);                    // [ST][16][PITCH]
  T* as = ring_w + ST * NC * PITCH;                             // [ST][16][PITCH], or the 16 whole rows
  float* cs = reinterpret_cast<float*>(as + (stream_a ? ST * 16 * PITCH : 16 * apitch));   // [8][16][CP]
  const int per_head = p.hd >> 4, half = p.hd >> 1;
  const int units = epi == EPI_QKV ? (p.nq + 2 * p.nkv) * per_head : epi == EPI_SWIGLU ? (g.N + 7) / 8 : (g.N + NC - 1) / NC;
  const int MT = (g.M + 15) / 16;
  // a long K and few tiles: the two groups of a CTA take half of the chunks of one tile each
  const bool split = chunks > 1 && MT * units <= (int)gridDim.x;
  const int cb = split ? gr.id * (chunks / 2) : 0, ce = split && gr.id == 0 ? chunks / 2 : chunks;
  const int vid = split ? (int)blockIdx.x : gr.vid, nv = split ? (int)gridDim.x : gr.nv;
  const int per = MT <= nv ? nv / MT : 1;   // groups (CTAs) on a row tile
  bool waited = false;
#pragma unroll 1
  for (int mt = MT <= nv ? vid % MT : vid; !waited || mt < MT; mt += (MT <= nv ? MT : nv)) {
    const int first = MT <= nv ? vid / MT : 0, m0 = mt * 16;
    const int mine = (mt < MT && first < per && first < units) ? (units - first + per - 1) / per : 0;
    const int total = mine * (ce - cb);
    int iu = first, ic = cb, is = 0, issued = 0;   // next step to load: unit, chunk, ring slot
    // A thread copies one column piece of rows pr, pr + RS, .. of a chunk: of W the first eight rows and the other
    // eight are runs of their own (their partner features, or the same rows of the other matrix).
    auto issue = [&](bool with_w, bool with_a, int u, int c, int s) {
      const int t = afresh(gr.t), pr = t / PPR, pk = (t % PPR) * PIECE;   // this thread's piece of a chunk: row, column
      const int k0 = c * KC + pk, full = max(0, min(16, (g.K - k0) * (int)sizeof(T)));
      if (with_w) {
        const T *wa = g.w0, *wb = g.w0;
        int n = u * NC, run = 8, left = g.N - n;      // first row, the second run's distance, rows of the matrix from n on
        if (epi == EPI_QKV) {
          const int head = u / per_head;
          wa = head < p.nq ? g.w0 : head < p.nq + p.nkv ? g.w1 : g.w2;
          wb = wa;
          n = (head < p.nq ? head : head < p.nq + p.nkv ? head - p.nq : head - p.nq - p.nkv) * p.hd + (u - head * per_head) * 8;
          run = half; left = 8;
        } else if (epi == EPI_SWIGLU) {
          wb = g.w1; n = u * 8; run = 0; left = g.N - n;
        }
        const int left_b = epi == EPI_STORE_F32 || epi == EPI_ADD_F32 ? left - 8 : left;
        wa += (size_t)(n + pr) * g.K + k0;
        wb += (size_t)(n + run + pr) * g.K + k0;
        T* dst = ring_w + ((size_t)s * NC + pr) * PITCH + pk;
#pragma unroll
        for (int i = 0; i < NP / 2; ++i) {
          const int r = i * RS;                       // row inside the run, from pr on
          const int ba = pr + r < left ? full : 0, bb = pr + r < left_b ? full : 0;
          cp_async16(dst + (size_t)r * PITCH, ba ? wa + (size_t)r * g.K : g.w0, ba);
          cp_async16(dst + (size_t)(r + 8) * PITCH, bb ? wb + (size_t)r * g.K : g.w0, bb);
        }
      }
      if (with_a && stream_a) {
        const T* src = g.A + (size_t)(m0 + pr) * g.K + k0;
        T* dst = as + ((size_t)s * 16 + pr) * PITCH + pk;
#pragma unroll
        for (int i = 0; i < NP; ++i) {
          const int bytes = m0 + pr + i * RS < g.M ? full : 0;
          cp_async16(dst + (size_t)i * RS * PITCH, bytes ? src + (size_t)i * RS * g.K : g.A, bytes);
        }
      }
    };
    const bool before = !waited;   // the weights of the first steps are on their way while the CTA waits
    if (!before) gsync(gr);        // the rows of the tile before have been read
#pragma unroll 1
    for (int pass = before ? 0 : 1; pass < 2; ++pass) {
      if (pass == 1 && before) {
        if (!wait()) return false;
        waited = true;
      }
      iu = first; ic = cb; is = 0; issued = 0;
#pragma unroll 1
      for (int s = 0; s < ST - 1; ++s) {
        if (issued < total) {
          issue(pass == 0 || !before, pass == 1, iu, ic, is);
          if (++ic == ce) { ic = cb; iu += per; }
          ++is; ++issued;
        }
        if (pass == 1) asm volatile("cp.async.commit_group;" ::: "memory");
      }
    }
    if (total == 0) continue;
    if (!stream_a) {
      const int r = gr.warp * 2 + (gr.lane >> 4), row = m0 + r;
      T* dst = as + (size_t)r * apitch;
      const float* xr = nullptr;
      T *g0 = nullptr, *g1 = nullptr;
      const int l = afresh(gr.lane & 15);
      bool norm = true;
      if (g.src == SRC_LM) norm = lm_row<T>(p, row, dst, chunks * KC, first == 0, l, xr, g0, g1);
      else if (row < g.M) xr = p.x + (size_t)row * p.d;
      if (__any_sync(0xffffffffu, norm || g1 != nullptr))       // both halves of the warp take part
        norm_row<T>(xr, g.gain, p.eps, p.d, norm ? dst : nullptr, chunks * KC, g0, g1, l);
    }
    f2 acc[4][4];
    float old = 0.f;             // residual value that the epilogue adds to
    int u = first, c = cb, slot = 0;
#pragma unroll 1
    for (int step = 0; step < total; ++step) {
      asm volatile("cp.async.wait_group %0;" ::"n"(ST - 2) : "memory");
      gsync(gr);                 // this step's chunk has landed for every thread; the slot of the last one is free
      if (issued < total) {
        issue(true, true, iu, ic, is);
        if (++ic == ce) { ic = cb; iu += per; }
        if (++is == ST) is = 0;
        ++issued;
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
      const int er = gr.t >> 4, ec = gr.t & 15;                 // the epilogue's element of this thread
      if (c == cb) {
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = 0ull;
        if (epi == EPI_ADD_F32 && m0 + er < g.M && u * NC + ec < g.N) old = __ldcg(g.C + (size_t)(m0 + er) * g.ldc + u * NC + ec);
      }
      // A warp has 32 k of a chunk, half of it 16 of them, a lane 4 x 4 outputs: rows ty + 4 i, columns tx + 4 j.  (What a
      // tile costs is the return path of its shared-memory loads, 4 clocks each: 32 a lane, and 48 with all 32 k in one
      // lane and 4 x 2 outputs.)
      const int t = afresh(gr.t), ty = (t >> 2) & 3, tx = t & 3, ko = (t >> 5) * (KC / 8) + ((t >> 4) & 1) * (KC / 16);
      const T* wp = ring_w + ((size_t)slot * NC + tx) * PITCH + ko;
      const T* ap = (stream_a ? as + (size_t)slot * 16 * PITCH : as + c * KC) + ty * apitch + ko;
#pragma unroll 1
      for (int k = 0; k < KC / 16; k += 4) {
        f2 wv[4][2];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          float v[4];
          load4<T>(wp + j * 4 * PITCH + k, v);
          wv[j][0] = pack2(v[0], v[1]); wv[j][1] = pack2(v[2], v[3]);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          float v[4];
          load4<T>(ap + i * 4 * apitch + k, v);
          const f2 a0 = pack2(v[0], v[1]), a1 = pack2(v[2], v[3]);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            fma2(acc[i][j], a0, wv[j][0]);
            fma2(acc[i][j], a1, wv[j][1]);
          }
        }
      }
      if (++slot == ST) slot = 0;
      if (++c < ce) continue;
      c = cb;
      // the two halves of the warp meet, each keeps two of the four rows
      const bool hi = gr.lane >= 16;
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float lo_v = sum2(acc[i][j]), hi_v = sum2(acc[i + 2][j]);
          const float got = __shfl_xor_sync(0xffffffffu, hi ? lo_v : hi_v, 16);
          cs[(gr.warp * 16 + ty + 4 * (i + (hi ? 2 : 0))) * CP + tx + 4 * j] = (hi ? hi_v : lo_v) + got;
        }
      float y = 0.f;
      if (split) {     // (one tile per CTA, so the sums are not overwritten)
        asm volatile("bar.sync 3, %0;" ::"n"(kFuseThreads) : "memory");
        if (gr.id != 0) break;
        const float* ct = cs + p.group_smem / (int)sizeof(float);
#pragma unroll
        for (int w = 0; w < 8; ++w) y += ct[(w * 16 + er) * CP + ec];
      } else {
        gsync(gr);
      }
#pragma unroll
      for (int w = 0; w < 8; ++w) y += cs[(w * 16 + er) * CP + ec];
      const int m = m0 + er;
      if (epi <= EPI_ADD_F32) {
        if (m < g.M && u * NC + ec < g.N) g.C[(size_t)m * g.ldc + u * NC + ec] = epi == EPI_ADD_F32 ? old + y : y;
      } else {
        const float y2 = __shfl_down_sync(0xffffffffu, y, 8);   // the partner feature's column
        if (ec < 8 && m < g.M) {
          if (epi == EPI_SWIGLU) {
            const int f = u * 8 + ec;
            if (f < g.N) g.act[(size_t)m * g.N + f] = from_f<T>(y / (1.f + expf(-y)) * y2);
          } else {
            const int head = u / per_head;
            simt_store_qkv<T>(qv, m, head, (u - head * per_head) * 8 + ec, y, y2);
          }
        }
      }
      u += per;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
  }
  return true;
}

// Bidirectional attention: a unit is 4 query rows of one head and variant, two warps per row with half of
// the keys of every tile each.  (It is bound by shared-memory reads, every warp reads its keys' K and V:
// with a row per warp and all keys a tile of 64 keys took 6300 clocks.)  Tiles of p.kt keys arrive in two
// buffers as they lie in memory (cached V transposed, active V row-major).
template <typename T, typename Wait>
__device__ bool attn_phase(const SimtStep<T>& p, int layer, const Group& gr, Wait&& wait) {
  constexpr int PIECE = GemmIo<T>::kPiece;
  const SeqMeta& m = p.m;
  const int hd = p.hd, kt = p.kt, kp = hd + PIECE, vp = kt + PIECE;
  const int vbuf = max(kt * kp, hd * vp);
  T* kb = reinterpret_cast<T*>(gr.smem);             // [2][kt][kp]
  T* vb = kb + 2 * kt * kp;                          // [2][vbuf]
  float* qs = reinterpret_cast<float*>(vb + 2 * vbuf) + gr.warp * (hd + 32);   // this warp's query row, then its probabilities
  float* ps = qs + hd;
  float* other = reinterpret_cast<float*>(vb + 2 * vbuf) + (gr.warp ^ 1) * (hd + 32);
  const int kw = kt / 2, kb0 = (gr.warp & 1) * kw;              // this warp's keys of a tile (32 or 16)
  const int nrt = (m.R_cap + 3) / 4, units = nrt * p.nq * m.nv * m.batch, ld = p.nkv * hd;
  const int hq = hd / PIECE, kj = gr.t / hq, kq0 = gr.t % hq;   // this thread's first piece of a K tile
  const float scale = rsqrtf((float)hd);
  bool waited = false;
#pragma unroll 1
  for (int unit = gr.vid; unit < units || !waited; unit += gr.nv) {
    const bool has = unit < units;
    const int vbi = unit / (nrt * p.nq), rem = unit - vbi * nrt * p.nq, h = rem / nrt, r0 = (rem - h * nrt) * 4;
    const int b = has ? vbi % m.batch : 0, vv = vbi / m.batch;
    const int P = m.ctx_len[b], R = m.last_len[b] + m.win_len[b], kvh = h / (p.nq / p.nkv);
    const int row0 = act_row(m, vv, b, 0);
    const int tc = (P + kt - 1) / kt, nt = (has && r0 < R) ? tc + (R + kt - 1) / kt : 0;
    const size_t kv = (size_t)layer * p.cache_layer + ((size_t)b * p.nkv + kvh) * (size_t)p.max_ctx * hd;
    auto load = [&](int t) {
      if (t < nt) {
        const bool ctx = t < tc;
        const int j0 = (ctx ? t : t - tc) * kt, n = min(kt, (ctx ? P : R) - j0);
        T* kd = kb + (size_t)(t & 1) * kt * kp;
        T* vd = vb + (size_t)(t & 1) * vbuf;
#pragma unroll 1
        for (int j = kj, q = kq0; j < kt; j += 256 / hq, q += 256 % hq) {
          if (q >= hq) { q -= hq; if (++j >= kt) break; }
          const int e = q * PIECE;
          const T* src = ctx ? p.k_cache + kv + (size_t)(j0 + j) * hd + e : p.k + (size_t)(row0 + j0 + j) * ld + kvh * hd + e;
          cp_async16(kd + j * kp + e, j < n ? src : p.k, j < n ? 16 : 0);
          if (!ctx) {
            const T* vs = p.v + (size_t)(row0 + j0 + j) * ld + kvh * hd + e;
            cp_async16(vd + j * kp + e, j < n ? vs : p.v, j < n ? 16 : 0);
          }
        }
        if (ctx) {   // keys are contiguous; what the cache holds beyond ctx_len is not read
          const int kq = kt / PIECE;
#pragma unroll 1
          for (int e = gr.t / kq; e < hd; e += 256 / kq) {   // kq is a power of two
            const int j = (gr.t % kq) * PIECE, bytes = max(0, min(16, (n - j) * (int)sizeof(T)));
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
    const int row = r0 + (gr.warp >> 1);
    const bool live = row < R;
    if (live)
      for (int e = gr.lane * 4; e < hd; e += 128) {
        float v[4];
        ldcg4<T>(p.q + (size_t)(row0 + row) * p.nq * hd + (size_t)h * hd + e, v);
        *reinterpret_cast<float4*>(qs + e) = make_float4(v[0], v[1], v[2], v[3]);
      }
    float mx = -INFINITY, sum = 0.f, o[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
    for (int t = 0; t < nt; ++t) {
      load(t + 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
      gsync(gr);
      if (live) {
        const bool ctx = t < tc;
        const int n = min(kt, ctx ? P - t * kt : R - (t - tc) * kt);
        const T* kd = kb + (size_t)(t & 1) * kt * kp;
        const T* vd = vb + (size_t)(t & 1) * vbuf;
        const int key = kb0 + gr.lane;                          // one key per lane
        const bool mine = gr.lane < kw && key < n;
        const T* kr = kd + (gr.lane < kw ? key : kb0) * kp;
        float a0 = 0.f, a1 = 0.f;
#pragma unroll 4
        for (int e = 0; e < hd; e += 4) {
          float x[4];
          load4<T>(kr + e, x);
          const float4 qv = *reinterpret_cast<const float4*>(qs + e);
          a0 = fmaf(qv.x, x[0], a0); a1 = fmaf(qv.y, x[1], a1); a0 = fmaf(qv.z, x[2], a0); a1 = fmaf(qv.w, x[3], a1);
        }
        const float s0 = mine ? (a0 + a1) * scale : -INFINITY;
        const float nm = fmaxf(mx, warp_max(s0));
        // (a warp may have no valid key so far: its reference point is still -inf, its sums are 0)
        const float corr = nm > -INFINITY ? expf(mx - nm) : 1.f, e0 = mine ? expf(s0 - nm) : 0.f;
        __syncwarp();
        ps[gr.lane] = e0;
        sum = sum * corr + warp_sum(e0);
        mx = nm;
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 4; ++i) o[i] *= corr;
        // features lane, lane + 32, ..: cached V has the keys contiguous, active V the features
        const T* vr = ctx ? vd + gr.lane * vp + kb0 : vd + kb0 * kp + gr.lane;
#pragma unroll 2
        for (int j = 0; j < kw; j += 4) {
          const float4 pv = *reinterpret_cast<const float4*>(ps + j);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            if (32 * i >= hd) break;
            float w[4];
            if (ctx) load4<T>(vr + 32 * i * vp + j, w);
            else {
#pragma unroll
              for (int c = 0; c < 4; ++c) w[c] = to_f<T>(vr[(j + c) * kp + 32 * i]);
            }
            o[i] = fmaf(pv.x, w[0], o[i]); o[i] = fmaf(pv.y, w[1], o[i]); o[i] = fmaf(pv.z, w[2], o[i]); o[i] = fmaf(pv.w, w[3], o[i]);
          }
        }
      }
      gsync(gr);
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    // the two halves of a row meet: the odd warp leaves its sums where its query row was
    if (gr.warp & 1) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (32 * i < hd) qs[gr.lane + 32 * i] = o[i];
      if (gr.lane == 0) { ps[0] = mx; ps[1] = sum; }
    }
    gsync(gr);
    if (live && !(gr.warp & 1)) {
      const float m2 = other[hd], s2 = other[hd + 1], top = fmaxf(mx, m2);
      const float c1 = expf(mx - top), c2 = m2 > -INFINITY ? expf(m2 - top) : 0.f;   // (this warp has the first key)
      const float inv = 1.f / (sum * c1 + s2 * c2);
      T* dst = p.o + (size_t)(row0 + row) * p.nq * hd + (size_t)h * hd;
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (32 * i < hd) dst[gr.lane + 32 * i] = from_f<T>((o[i] * c1 + other[gr.lane + 32 * i] * c2) * inv);
    }
    gsync(gr);
  }
  return true;
}

// Cross log-probs (Eq. 6 halves): xlogp[b,i,j] = h_i . W_lm[yhat_j] - lse_i.  A unit is a column j and 16
// rows, two per warp.
template <typename T>
__device__ __forceinline__ void xlogp_phase(const SimtStep<T>& p, const Group& gr) {
  const SeqMeta& m = p.ml;
  const int it = (m.W_cap + 15) / 16, units = m.batch * m.W_cap * it;
  for (int unit = gr.vid; unit < units; unit += gr.nv) {
    const int bj = unit / it, b = bj / m.W_cap, j = bj - b * m.W_cap, W = m.win_len[b];
    if (j >= W) continue;
    const int tok = __ldcg(p.sig.ws_pred + b * m.W_cap + j);
    const bool ok = tok >= 0 && tok < p.V;   // never index the vocabulary matrix with an id outside it
    const T* wr = p.lm_head + (size_t)(ok ? tok : 0) * p.d;
    const int i0 = (unit - bj * it) * 16 + gr.warp * 2;
    if (i0 >= W) continue;
    const bool two = i0 + 1 < W;
    const T* h0 = p.h + (size_t)lm_row(m, 0, b * m.W_cap + i0) * p.d;
    const T* h1 = p.h + (size_t)lm_row(m, 0, b * m.W_cap + i0 + (two ? 1 : 0)) * p.d;
    float a0 = 0.f, a1 = 0.f;
#pragma unroll 2
    for (int e = gr.lane * 4; e < p.d; e += 128) {
      float w[4], x[4], y[4];
      load4<T>(wr + e, w);
      ldcg4<T>(h0 + e, x);
      ldcg4<T>(h1 + e, y);
#pragma unroll
      for (int c = 0; c < 4; ++c) { a0 = fmaf(x[c], w[c], a0); a1 = fmaf(y[c], w[c], a1); }
    }
    a0 = warp_sum(a0); a1 = warp_sum(a1);
    if (gr.lane < (two ? 2 : 1)) {
      const int i = i0 + gr.lane;
      p.xlogp[((size_t)b * p.max_window + i) * p.max_window + j] =
          ok ? (gr.lane ? a1 : a0) - __ldcg(p.sig.ws_lse + b * m.W_cap + i) : -INFINITY;
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
    if (go == 0) asm volatile("cp.async.wait_all;" ::: "memory");   // the copies that the next phase had under way
    return go != 0;
  };
  if (p.stall && blockIdx.x == 0) return;

  const int M = p.m.nv * p.m.rows, n_phases = 5 * p.n_layers;
#pragma unroll 1
  for (int ph = 0; ph <= n_phases; ++ph) {
    const int l = ph / 5, kind = ph == n_phases ? 5 : ph - 5 * l;   // QKV, attention, O, gate / up, down; LM head
    if (ph > 0) arrive();
    if (kind == 1) {
      if (!attn_phase<T>(p, l, gr, wait)) return;
      continue;
    }
    const SimtLayer<T>* L = p.layers + l;
    const size_t cache = (size_t)l * p.cache_layer;
    QkvView<T> qv{p.m, p.nq, p.nkv, p.hd, p.max_ctx, p.cos_sin, nullptr, nullptr, nullptr, p.q, p.k, p.v,
                  p.export_kv ? p.k_cache + cache : nullptr, p.export_kv ? p.v_cache + cache : nullptr};
    FuseGemm<T> g{nullptr, nullptr, nullptr, nullptr, nullptr, M, p.d, p.d, p.d, p.x, p.act, EPI_ADD_F32, SRC_GLOBAL};
    if (kind == 0) {
      g.w0 = L->wq; g.w1 = L->wk; g.w2 = L->wv; g.gain = L->n1; g.epi = EPI_QKV; g.src = SRC_NORM;
      qv.bq = L->bq; qv.bk = L->bk; qv.bv = L->bv;
    } else if (kind == 2) {
      g.A = p.o; g.w0 = L->wo; g.K = p.nq * p.hd;
    } else if (kind == 3) {
      g.w0 = L->wg; g.w1 = L->wu; g.gain = L->n2; g.N = p.F; g.epi = EPI_SWIGLU; g.src = SRC_NORM;
    } else if (kind == 4) {
      g.A = p.act; g.w0 = L->wd; g.K = p.F;
    } else {
      g.w0 = p.lm_head; g.gain = p.final_norm; g.M = p.ml.nv * p.ml.npos_pad; g.N = p.V; g.C = p.logits; g.ldc = p.V;
      g.epi = EPI_STORE_F32; g.src = SRC_LM;
    }
    if (!gemm_phase<T>(p, g, qv, gr, wait)) return;
    if (p.kv_only && ph == n_phases - 5) return;   // prefill: nothing after the last layer's K / V is used
  }
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
      if (p.max_window <= 64) boundary_seq<2, 1, true>(p.sig.ws_infl, p.sig.ws_ent, b, p.ml, DevLens{}, p.hp, p.bnd, bnd[0], bnd[1]);
      else boundary_seq<DC_MAX_WINDOW / 32, 1, true>(p.sig.ws_infl, p.sig.ws_ent, b, p.ml, DevLens{}, p.hp, p.bnd, bnd[0], bnd[1]);
}

template <typename T>
size_t group_smem(int d, int hd, int kt) {
  const size_t pitch = kKC + GemmIo<T>::kPad, rows = (size_t)(d + kKC - 1) / kKC * kKC + GemmIo<T>::kPad;
  const size_t gemm = 16 * (kStages * pitch + (kStages * pitch > rows ? kStages * pitch : rows)) * sizeof(T) + 8 * 16 * 17 * sizeof(float);
  const size_t kp = hd + GemmIo<T>::kPiece, vp = kt + GemmIo<T>::kPiece;
  const size_t vb = kt * kp > hd * vp ? kt * kp : hd * vp;
  const size_t attn = 2 * (kt * kp + vb) * sizeof(T) + 8 * (size_t)(hd + 32) * sizeof(float);
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
  // the answer is the device's, not the context's: asked once (a racing context finds the same)
  static std::atomic<int> sms_of[64];
  int dev = 0, sms = 0, coop = 0;
  cudaGetDevice(&dev);
  if (dev < 64) sms = sms_of[dev].load(std::memory_order_acquire);
  if (sms == 0) {
    cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    int per_sm = 0;
    if (cudaFuncSetAttribute(k_simt_step<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kGroups * kGroupSmemMax)) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_simt_step<T>, kFuseThreads, kGroups * kGroupSmemMax) != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    if (!coop || sms < 1 || per_sm < 1) sms = -1;
    if (dev < 64) sms_of[dev].store(sms, std::memory_order_release);
  }
  if (sms > 0) f->grid = sms;
  return true;
}

template <typename T>
bool simt_step_ok(const SimtFuse& f, const SimtStep<T>& p) {
  if (f.grid == 0) return false;
  // GEMMs that take many rounds of small tiles are better off as kernels of their own, with the larger tile
  const long long M = (long long)p.m.nv * p.m.rows, Mlm = (long long)p.ml.nv * p.ml.npos_pad;
  const long long mt = (M + 15) / 16;
  long long most = mt * ((p.F + 7) / 8);
  const long long qkv = mt * (p.nq + 2 * p.nkv) * (p.hd / 16), lm = p.kv_only ? 0 : (Mlm + 15) / 16 * ((p.V + 15) / 16);
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
