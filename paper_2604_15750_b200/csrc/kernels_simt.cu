// CUDA-core kernels of the block-step: any shape, fp32 or bf16 storage, fp32 arithmetic.
// They are the whole path for fp32 models and for shapes the tensor-core kernels do not take,
// and the small glue kernels (embedding gather, norms, RoPE, SwiGLU, signals, cross log-probs)
// of the tensor-core path.
#include <math.h>

#include <atomic>
#include <type_traits>

#include "pdl.cuh"
#include "simt_dev.cuh"

namespace dc {

constexpr size_t kSimtSmemMax = 220 * 1024;   // dynamic shared memory a kernel of this file may ask for

// block-wide sum for blockDim.x <= 1024 (multiple of 32); red: >= 32 floats of shared memory
__device__ __forceinline__ float block_sum(float v, float* red) {
  v = warp_sum(v);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = blockDim.x >> 5;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  float t = (l < nw) ? red[l] : 0.f;
  t = warp_sum(t);
  return t;
}

// ---- start of a step: embedding gather, RoPE table, cleared words -----------------------------------
// Blocks [0, M): x[row] = E[token of row].  Variant 0 (curr): [last block ; window]; variant 1 (prev):
// the last block's ids replaced by the mask id, everything else fixed, which makes p_prev =
// p(Z_k | c) (Section 4.4).  The block of a sequence's first curr row checks all of its ids and writes
// status[b] (so that nothing has to clear it first).
// The other blocks: cos_sin[(row0[b] + r) * hd + i] = cos(angle), [.. + hd/2 + i] = sin(angle), angle =
// (pos0[b] + r) * theta^(-2i/hd), evaluated in double precision; row `rows` holds cos / sin of
// theta^(-2i/hd) itself, the angle step between consecutive rows.  The first of them also clears the
// grid-barrier words of the kernels that follow.
// (One launch: as a memset and two kernels the start of a step took 8 us, most of it launch latency.)
template <typename T>
__global__ void __launch_bounds__(128) k_step_begin(const T* __restrict__ embed, const int32_t* __restrict__ last_ids,
                                                    const int32_t* __restrict__ win_ids, int max_last, int max_window,
                                                    int mask_id, int vocab, int d, const __grid_constant__ SeqMeta m,
                                                    float* __restrict__ x, int32_t* __restrict__ status, int hd, float theta,
                                                    float* __restrict__ cos_sin, unsigned int* __restrict__ words, int n_words) {
  pdl_trigger();
  const int M = m.nv * m.rows, row = blockIdx.x;
  if (row < M) {
    const int v = row / m.rows, br = row - v * m.rows, b = act_seq(m, br), r = br - m.row0[b];
    const int Lb = m.last_len[b], W = m.win_len[b];
    if (r == 0 && v == 0) {
      int bad = 0;
      for (int i = threadIdx.x; i < Lb + W; i += blockDim.x) {
        const int id = i < Lb ? last_ids[b * max_last + i] : win_ids[b * max_window + i - Lb];
        bad |= (id < 0 || id >= vocab);
      }
      bad = __syncthreads_or(bad);
      if (threadIdx.x == 0) status[b] = bad ? DC_ERR_INDEX : DC_OK;
    }
    int tok = mask_id;
    if (r < Lb) tok = (v == 0) ? last_ids[b * max_last + r] : mask_id;
    else if (r < Lb + W) tok = win_ids[b * max_window + (r - Lb)];
    if (tok < 0 || tok >= vocab) tok = mask_id;
    const T* e = embed + (size_t)tok * d;
    float* xr = x + (size_t)row * d;
    // d is a multiple of 4: four elements per thread and step
#pragma unroll 8
    for (int i = threadIdx.x * 4; i < d; i += 128 * 4) {
      float w[4];
      load4<T>(e + i, w);
      *reinterpret_cast<float4*>(xr + i) = make_float4(w[0], w[1], w[2], w[3]);
    }
    return;
  }
  if (row == M)
    for (int i = threadIdx.x; i < n_words; i += blockDim.x) words[i] = 0u;
  const int half = hd / 2;
  const int idx = (row - M) * 128 + threadIdx.x;
  const int rows = m.rows;
  if (idx >= (rows + 1) * half) return;   // one extra row: cos / sin of the per-row angle step
  const int i = idx % half, br = idx / half;
  const int b = act_seq(m, br), r = br - m.row0[b];
  const double inv_freq = pow((double)theta, -2.0 * (double)i / (double)hd);
  const double ang = (br < rows) ? (double)(m.pos0[b] + r) * inv_freq : inv_freq;
  double sn, cs;
  sincos(ang, &sn, &cs);
  cos_sin[(size_t)br * hd + i] = (float)cs;
  cos_sin[(size_t)br * hd + half + i] = (float)sn;
}

// (An ordinary launch: what comes before the step in the stream has completed when it starts.  The GEMMs' early weight
// loads rely on that: pdl.cuh.)
template <typename T>
void launch_step_begin(const T* embed, const int32_t* last_ids, const int32_t* win_ids, int max_last, int max_window,
                       int mask_id, int vocab, int d, const SeqMeta& m, float* x, int32_t* status, int head_dim,
                       float theta, float* cos_sin, unsigned int* words, int n_words, cudaStream_t s) {
  const int M = m.nv * m.rows, table = (m.rows + 1) * (head_dim / 2);
  k_step_begin<T><<<M + (table + 127) / 128, 128, 0, s>>>(embed, last_ids, win_ids, max_last, max_window, mask_id, vocab,
                                                          d, m, x, status, head_dim, theta, cos_sin, words, n_words);
}

// ---- RMSNorm (with the split-K partial sums of the preceding GEMM folded into x) --------------
// One row per block; d is a multiple of 4.  The row (with the partial sums folded in, in split
// order, so the result does not depend on the launch shape) is written back to x and normed.
// (The partial sums as constant data, so that their loads may pass the stores to x: 1.2% of a step of four Dream-7B
// sequences.  The pointer has gone through the wait for the kernel that wrote them.)
template <typename T>
__device__ __forceinline__ void rmsnorm_row(float* __restrict__ xr, const float* __restrict__ part,
                                            int nsplit, size_t part_stride, const T* __restrict__ g,
                                            float eps, int d, T* __restrict__ outr, float* red) {
  float ss = 0.f;
  for (int i = threadIdx.x * 4; i < d; i += blockDim.x * 4) {
    float4 v = *reinterpret_cast<const float4*>(xr + i);
    if (part) {
      for (int sidx = 0; sidx < nsplit; ++sidx) {
        const float4 pv = __ldg(reinterpret_cast<const float4*>(part + sidx * part_stride + i));
        v.x += pv.x; v.y += pv.y; v.z += pv.z; v.w += pv.w;
      }
      *reinterpret_cast<float4*>(xr + i) = v;
    }
    ss += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
  }
  ss = block_sum(ss, red);
  const float inv = rsqrtf(ss / (float)d + eps);
  for (int i = threadIdx.x * 4; i < d; i += blockDim.x * 4) {
    const float4 v = *reinterpret_cast<const float4*>(xr + i);
    float gv[4];
    load4<T>(g + i, gv);
    const float o[4] = {v.x * inv * gv[0], v.y * inv * gv[1], v.z * inv * gv[2], v.w * inv * gv[3]};
    store4<T>(outr + i, o);
  }
}

// The same with the row in registers, NI pieces of four a thread: all loads of x and of the partial sums are under way at
// once, where a piece after the other is a chain of 2 NI memory latencies (the loads of x may not pass its stores).
template <typename T, int NI>
__device__ __forceinline__ void rmsnorm_row_regs(float* __restrict__ xr, const float* __restrict__ part,
                                                 int nsplit, size_t part_stride, const T* __restrict__ g,
                                                 float eps, int d, T* __restrict__ outr, float* red) {
  float4 v[NI];
  const int t4 = threadIdx.x * 4;
#pragma unroll
  for (int k = 0; k < NI; ++k)
    v[k] = t4 + k * 1024 < d ? *reinterpret_cast<const float4*>(xr + t4 + k * 1024) : make_float4(0.f, 0.f, 0.f, 0.f);
  if (part) {
#pragma unroll 2
    for (int sidx = 0; sidx < nsplit; ++sidx) {
      const float* ps = part + sidx * part_stride;
      float4 w[NI];
#pragma unroll
      for (int k = 0; k < NI; ++k)
        w[k] = t4 + k * 1024 < d ? __ldg(reinterpret_cast<const float4*>(ps + t4 + k * 1024)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int k = 0; k < NI; ++k) { v[k].x += w[k].x; v[k].y += w[k].y; v[k].z += w[k].z; v[k].w += w[k].w; }
    }
  }
  float gv[NI][4];
#pragma unroll
  for (int k = 0; k < NI; ++k)
    if (t4 + k * 1024 < d) load4<T>(g + t4 + k * 1024, gv[k]);
  float ss = 0.f;
#pragma unroll
  for (int k = 0; k < NI; ++k) {
    if (part && t4 + k * 1024 < d) *reinterpret_cast<float4*>(xr + t4 + k * 1024) = v[k];
    ss += v[k].x * v[k].x + v[k].y * v[k].y + v[k].z * v[k].z + v[k].w * v[k].w;
  }
  ss = block_sum(ss, red);
  const float inv = rsqrtf(ss / (float)d + eps);
#pragma unroll
  for (int k = 0; k < NI; ++k)
    if (t4 + k * 1024 < d) {
      const float o[4] = {v[k].x * inv * gv[k][0], v[k].y * inv * gv[k][1], v[k].z * inv * gv[k][2], v[k].w * inv * gv[k][3]};
      store4<T>(outr + t4 + k * 1024, o);
    }
}

template <typename T, int NI>   // NI: pieces of 1024 elements of a row, 0: any width
__global__ void __launch_bounds__(256) k_rmsnorm(float* __restrict__ x,
                                                 const float* __restrict__ part, int nsplit,
                                                 size_t part_stride, const T* __restrict__ g,
                                                 float eps, int d, T* __restrict__ out) {
  __shared__ float red[32];
  pdl_trigger();
  pdl_wait(x, part);
  const size_t off = (size_t)blockIdx.x * d;
  if constexpr (NI > 0)
    rmsnorm_row_regs<T, NI>(x + off, part ? part + off : nullptr, nsplit, part_stride, g, eps, d, out + off, red);
  else
    rmsnorm_row<T>(x + off, part ? part + off : nullptr, nsplit, part_stride, g, eps, d, out + off, red);
}

template <typename T>
void launch_rmsnorm(float* x, const float* part, int nsplit, size_t part_stride, const T* g,
                    float eps, int M, int d, T* out, cudaStream_t s) {
  auto* k = d <= 1024 ? k_rmsnorm<T, 1> : d <= 2048 ? k_rmsnorm<T, 2> : d <= 4096 ? k_rmsnorm<T, 4> : d <= 8192 ? k_rmsnorm<T, 8> : k_rmsnorm<T, 0>;
  launch_chained(k, M, 256, 0, s, x, part, nsplit, part_stride, g, eps, d, out);
}

// LM-head input rows, one block per row of the LM head's order (groups of G positions: curr rows, then
// prev rows): the final norm of the window's rows (nothing reads x after it, so the folded row stays
// on chip); rows of p_prev carried in from an earlier step, or - no earlier prediction for the
// position - a copy of the curr row, which makes the two distributions equal and I_k = 0; the
// caller's shaped rows in place of either; and the copy of the curr rows that a later step carries.
// (One launch: as three the second and third cost 3 us each of a step for a few hundred KB.)
template <typename T>
__global__ void __launch_bounds__(256) k_lm_rows(const float* __restrict__ x, const float* __restrict__ part, int nsplit,
                                                 size_t part_stride, const T* __restrict__ g, float eps, int d,
                                                 const SeqMeta m, int nv_x, const LmRowsIo<T> io, T* __restrict__ h,
                                                 int staged) {
  extern __shared__ __align__(16) float lm_row_s[];   // staged: the row with the partial sums folded in
  __shared__ float red[32];
  pdl_trigger();
  pdl_wait(x, part);
  const int lrow = blockIdx.x;
  const int grp = lrow / (m.nv * m.G), in = lrow % (m.nv * m.G);
  const int v = in / m.G, p = grp * m.G + in % m.G;
  const int b = p / m.W_cap, k = p % m.W_cap;
  T* hr = h + (size_t)lrow * d;
  const T* src = nullptr;        // copied instead of normed
  bool norm = true;
  if (b >= m.batch || k >= m.win_len[b]) {
    norm = false;                // pad row: zero
  } else if (io.h_in != nullptr) {
    src = io.h_in + (((size_t)b * 2 + v) * io.max_window + k) * d;
    norm = v == 0 && io.h_out != nullptr;
  } else if (v >= nv_x && k < io.prev.n[b]) {
    src = io.h_prev_in + ((size_t)b * io.max_window + k) * d;
    norm = false;
  }
  if (src != nullptr || !norm) {
    for (int i = threadIdx.x * 4; i < d; i += blockDim.x * 4) {
      float o[4] = {0.f, 0.f, 0.f, 0.f};
      if (src != nullptr) load4<T>(src + i, o);
      store4<T>(hr + i, o);
    }
    if (!norm) return;
  }
  const size_t off = (size_t)act_row(m, v < nv_x ? v : 0, b, m.last_len[b] + k) * d;
  T* dst0 = src == nullptr ? hr : nullptr;
  T* dst1 = (v == 0 && io.h_out != nullptr) ? io.h_out + ((size_t)b * io.max_window + k) * d : nullptr;
  auto folded = [&](int i) {
    float4 w = *reinterpret_cast<const float4*>(x + off + i);
    if (part)
      for (int sidx = 0; sidx < nsplit; ++sidx) {
        const float4 pv = *reinterpret_cast<const float4*>(part + sidx * part_stride + off + i);
        w.x += pv.x; w.y += pv.y; w.z += pv.z; w.w += pv.w;
      }
    return w;
  };
  float ss = 0.f;
  for (int i = threadIdx.x * 4; i < d; i += blockDim.x * 4) {
    const float4 w = folded(i);
    if (staged) *reinterpret_cast<float4*>(lm_row_s + i) = w;
    ss += w.x * w.x + w.y * w.y + w.z * w.z + w.w * w.w;
  }
  ss = block_sum(ss, red);
  const float inv = rsqrtf(ss / (float)d + eps);
  for (int i = threadIdx.x * 4; i < d; i += blockDim.x * 4) {
    const float4 w = staged ? *reinterpret_cast<const float4*>(lm_row_s + i) : folded(i);
    float gv[4];
    load4<T>(g + i, gv);
    const float o[4] = {w.x * inv * gv[0], w.y * inv * gv[1], w.z * inv * gv[2], w.w * inv * gv[3]};
    if (dst0) store4<T>(dst0 + i, o);
    if (dst1) store4<T>(dst1 + i, o);
  }
}

template <typename T>
void launch_lm_rows(const float* x, const float* part, int nsplit, size_t part_stride, const T* g, float eps, int d,
                    const SeqMeta& m, int nv_x, const LmRowsIo<T>& io, T* h, cudaStream_t s) {
  // rows of more than 12256 elements are folded twice instead of staged: they have no room in the 48 KB that a
  // kernel may use without an opt-in (and 128 bytes are the sums')
  const size_t row = d * sizeof(float);
  const int staged = row + 128 <= 48 * 1024;
  launch_chained(k_lm_rows<T>, m.nv * m.npos_pad, 256, staged ? row : 0, s, x, part, nsplit, part_stride, g, eps, d, m, nv_x, io, h,
                 staged);
}

// ---- CUDA-core GEMM: acc[m, n] = sum_k A[m, k] W[n, k], fp32 FMAs, with the epilogues of a layer ----
//
// These run for models of a few million parameters (fp32, or shapes the tensor cores do not take),
// where a GEMM is 10..400 M FMAs and its time is the latency of one pass: load, multiply, reduce,
// store.  So the tile is small (16 x 32: 48..512 CTAs at d 256 instead of 4..64 with 64 x 64), the
// eight warps of a CTA split K among them (a chunk of 128 k is 16 per warp), chunks arrive through
// a three-stage cp.async ring, and a lane's 4 x 4 outputs are fed by 16-byte shared-memory reads of
// four k at a time, multiplied as packed fp32 pairs.  Measured with d 256, d_ff 1024, M 96 (a 64 x 64
// tile with element-wise loads before): QKV with its rotation 3 launches of 38 us + 2.3 -> 4.9 us,
// gate / up with SwiGLU 2 x 41 + 2 -> 7.3 us, O and down projection 41 -> 7.4 us on average.  Above
// kSmallTiles tiles (eight per SM) the 64 x 64 tile takes over: the same inner loop (bound by
// shared-memory reads either way) with a third of the L2 traffic per output, which binds once every
// SM holds several small tiles.
//
// A tile's 32 columns are either 32 consecutive rows of W, or - for the epilogues that combine two
// output features - 16 features and their partners: i and i + head_dim / 2 of a head (RoPE), or
// gate and up of an MLP feature.
template <typename T, int WM, int WN, int WK, int KC, int STAGES, int EPI>
__global__ void __launch_bounds__(256) k_gemm_simt(const SimtGemm<T> g) {
  constexpr int BM = 16 * WM, BN = 32 * WN, PITCH = KC + GemmIo<T>::kPad, PIECE = GemmIo<T>::kPiece;
  constexpr int ROWS = BM + BN, STAGE = ROWS * PITCH, CP = BN + 1;
  static_assert(WM * WN * WK == 8 && KC % (4 * WK) == 0 && KC % PIECE == 0, "eight warps");
  extern __shared__ __align__(16) unsigned char simt_smem[];
  T* ring = reinterpret_cast<T*>(simt_smem);
  float* cs = reinterpret_cast<float*>(simt_smem);     // [WK][BM][CP], over the ring once it is drained
  __shared__ const T* rowp[ROWS];                      // source rows of the tile; null: beyond the matrix
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int m0 = blockIdx.y * BM, u0 = blockIdx.x * WN;   // u: unit of 32 columns
  for (int r = tid; r < ROWS; r += 256) {
    const T* src = nullptr;
    if (r < BM) {
      if (m0 + r < g.M) src = g.A + (size_t)(m0 + r) * g.K;
    } else {
      const int j = r - BM, u = u0 + (j >> 5), jj = j & 31;
      if (EPI == EPI_QKV) {
        const int half = g.hd >> 1, per_head = g.hd >> 5, head = u / per_head;
        const int e = (u - head * per_head) * 16 + (jj & 15) + (jj >> 4) * half;
        if (head < g.nq) src = g.w0 + (size_t)(head * g.hd + e) * g.K;
        else if (head < g.nq + g.nkv) src = g.w1 + (size_t)((head - g.nq) * g.hd + e) * g.K;
        else if (head < g.nq + 2 * g.nkv) src = g.w2 + (size_t)((head - g.nq - g.nkv) * g.hd + e) * g.K;
      } else if (EPI == EPI_SWIGLU) {
        const int f = u * 16 + (jj & 15);
        if (f < g.N) src = (jj < 16 ? g.w0 : g.w1) + (size_t)f * g.K;
      } else {
        const int n = u * 32 + jj;
        if (n < g.N) src = g.w0 + (size_t)n * g.K;
      }
    }
    rowp[r] = src;
  }
  __syncthreads();

  const int chunks = (g.K + KC - 1) / KC;
  auto load = [&](int c) {
    T* dst = ring + (size_t)(c % STAGES) * STAGE;
    const int k0 = c * KC;
    if (g.vec) {
      for (int p = tid; p < ROWS * (KC / PIECE); p += 256) {
        const int r = p / (KC / PIECE), k = (p - r * (KC / PIECE)) * PIECE;
        const T* src = rowp[r];
        const int bytes = src == nullptr ? 0 : max(0, min(16, (g.K - k0 - k) * (int)sizeof(T)));
        cp_async16(dst + r * PITCH + k, bytes ? src + k0 + k : g.A, bytes);
      }
    } else {   // rows that are not 16-byte aligned
      for (int p = tid; p < ROWS * KC; p += 256) {
        const int r = p / KC, k = p - r * KC;
        const T* src = rowp[r];
        dst[r * PITCH + k] = (src != nullptr && k0 + k < g.K) ? src[k0 + k] : from_f<T>(0.f);
      }
    }
  };
  for (int c = 0; c < STAGES - 1; ++c) {
    if (c < chunks) load(c);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  const int wk = warp % WK, wn = (warp / WK) % WN, wm = warp / (WK * WN);
  const int ty = lane >> 3, tx = lane & 7;
  f2 acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
  for (int c = 0; c < chunks; ++c) {
    asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 2) : "memory");
    __syncthreads();     // chunk c has landed for every thread; the stage of chunk c - 1 is free
    if (c + STAGES - 1 < chunks) load(c + STAGES - 1);
    asm volatile("cp.async.commit_group;" ::: "memory");
    const T* st = ring + (size_t)(c % STAGES) * STAGE + wk * (KC / WK);
    const T* ap = st + (wm * 16 + ty * 4) * PITCH;
    const T* wp = st + (BM + wn * 32 + tx) * PITCH;
#pragma unroll
    for (int k = 0; k < KC / WK; k += 4) {
      f2 av[4][2], wv[4][2];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float v[4];
        load4<T>(ap + i * PITCH + k, v);
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
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();       // the ring is read; the sums go over it
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
      cs[(wk * BM + wm * 16 + ty * 4 + i) * CP + wn * 32 + tx + 8 * j] = sum2(acc[i][j]);
  __syncthreads();
  auto value = [&](int r, int c) {
    float v = cs[r * CP + c];
#pragma unroll
    for (int w = 1; w < WK; ++w) v += cs[(w * BM + r) * CP + c];
    return v;
  };
  if (EPI == EPI_STORE_F32 || EPI == EPI_ADD_F32) {
    for (int p = tid; p < BM * BN; p += 256) {
      const int r = p / BN, c = p - r * BN, m = m0 + r, n = u0 * 32 + c;
      if (m >= g.M || n >= g.N) continue;
      float* dst = g.C + (size_t)m * g.ldc + n;
      const float v = value(r, c);
      *dst = EPI == EPI_ADD_F32 ? *dst + v : v;
    }
  } else {
    for (int p = tid; p < BM * BN / 2; p += 256) {
      const int r = p / (BN / 2), c = p - r * (BN / 2), m = m0 + r;
      const int u = u0 + (c >> 4), i = c & 15;
      if (m >= g.M) continue;
      const float y1 = value(r, (c >> 4) * 32 + i), y2 = value(r, (c >> 4) * 32 + 16 + i);
      if (EPI == EPI_SWIGLU) {
        const int f = u * 16 + i;
        if (f < g.N) g.act[(size_t)m * g.N + f] = from_f<T>(y1 / (1.f + expf(-y1)) * y2);
      } else {
        const int half = g.hd >> 1, per_head = g.hd >> 5, head = u / per_head;
        if (head >= g.nq + 2 * g.nkv) continue;
        const int e = (u - head * per_head) * 16 + i;
        simt_store_qkv<T>(g, m, head, e, y1, y2);
      }
    }
  }
}

constexpr long long kSmallTiles = 148 * 8;

template <typename T, int EPI>
static void launch_gemm_epi(SimtGemm<T> g, int units, cudaStream_t s) {
  auto aligned = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
  g.vec = g.K % GemmIo<T>::kPiece == 0 && aligned(g.A) && aligned(g.w0) &&
          (g.w1 == nullptr || aligned(g.w1)) && (g.w2 == nullptr || aligned(g.w2));
  const long long tiles = (long long)((g.M + 15) / 16) * units;
  if (tiles <= kSmallTiles) {
    constexpr int KC = 128, STAGES = 3;
    const size_t ring = (size_t)STAGES * 48 * (KC + GemmIo<T>::kPad) * sizeof(T), sums = 8 * 16 * 33 * sizeof(float);
    k_gemm_simt<T, 1, 1, 8, KC, STAGES, EPI><<<dim3(units, (g.M + 15) / 16), 256, ring > sums ? ring : sums, s>>>(g);
  } else {
    constexpr int KC = 32, STAGES = 3;
    const size_t ring = (size_t)STAGES * 128 * (KC + GemmIo<T>::kPad) * sizeof(T), sums = 64 * 65 * sizeof(float);
    k_gemm_simt<T, 4, 2, 1, KC, STAGES, EPI><<<dim3((units + 1) / 2, (g.M + 63) / 64), 256, ring > sums ? ring : sums, s>>>(g);
  }
}

template <typename T>
void launch_gemm_simt(const SimtGemm<T>& g, int epi, cudaStream_t s) {
  switch (epi) {
    case EPI_STORE_F32: launch_gemm_epi<T, EPI_STORE_F32>(g, (g.N + 31) / 32, s); break;
    case EPI_ADD_F32: launch_gemm_epi<T, EPI_ADD_F32>(g, (g.N + 31) / 32, s); break;
    case EPI_SWIGLU: launch_gemm_epi<T, EPI_SWIGLU>(g, (g.N + 15) / 16, s); break;
    default: launch_gemm_epi<T, EPI_QKV>(g, (g.nq + 2 * g.nkv) * (g.hd / 32), s);
  }
}

// head_dim not a multiple of 32: the projections go through `tmp` [M, (nq + 2 nkv) hd] and this
// kernel, everything else has the rotation in the GEMM's epilogue.
template <typename T>
__global__ void k_rope_store(const float* __restrict__ tmp, const SimtGemm<T> g) {
  const int m = blockIdx.x, half = g.hd / 2, heads = g.nq + 2 * g.nkv;
  const float* t = tmp + (size_t)m * heads * g.hd;
  for (int idx = threadIdx.x; idx < heads * half; idx += blockDim.x) {
    const int head = idx / half, e = idx % half;
    simt_store_qkv<T>(g, m, head, e, t[head * g.hd + e], t[head * g.hd + half + e]);
  }
}

template <typename T>
void launch_rope_store(const float* tmp, const SimtGemm<T>& g, cudaStream_t s) {
  k_rope_store<T><<<g.M, 256, 0, s>>>(tmp, g);
}

// ---- bidirectional attention on CUDA cores ------------------------------------------------------
// Keys of query (v, b, r): the ctx_len[b] cached rows, then the last_len[b] + win_len[b] active
// rows of the same variant.  No causal mask.
//
// A CTA takes 16 query rows of one head (two per warp) and streams tiles of `kt` keys through
// shared memory with a running softmax: K rows and V columns are staged with padded pitches, so that
// a lane scores one key and accumulates one output feature with conflict-free 16-byte reads.  The
// work is tiny (a few MFMAs per head); what it took the time on was serial: one warp per row read
// every K row element by element from global memory (112 keys, head_dim 64: 44 -> 14 us).
constexpr int kAttnSimtRows = 16;
template <typename T>
__global__ void __launch_bounds__(256) k_attn_simt(
    const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ v,
    const T* __restrict__ k_cache, const T* __restrict__ v_cache, int max_ctx, const SeqMeta m, int nq,
    int nkv, int hd, T* __restrict__ o, int kt, int rows, int vec) {
  extern __shared__ __align__(16) float attn_smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int h = blockIdx.y, vb = blockIdx.z;
  const int b = vb % m.batch, vv = vb / m.batch;
  const int g = h / (nq / nkv);
  const int P = m.ctx_len[b], R = m.last_len[b] + m.win_len[b];
  const int r0 = blockIdx.x * rows;
  if (r0 >= R) return;
  const int hp = (hd + 3) / 4 * 4, kp = hp + 4, vp = kt + 4;   // padded head_dim; pitches of K and V^T rows
  float* Ks = attn_smem;                        // [kt][kp]
  float* Vs = Ks + (size_t)kt * kp;             // [hd][vp]
  float* qs = Vs + (size_t)hd * vp;             // [rows][kp]
  float* ps = qs + rows * kp;                   // [rows][vp]
  float* os = ps + rows * vp;                   // [rows][hp]
  const float scale = rsqrtf((float)hd);
  const size_t kvh = (size_t)b * nkv + g;
  const T* kc = k_cache ? k_cache + kvh * (size_t)max_ctx * hd : nullptr;
  const T* vc = v_cache ? v_cache + kvh * (size_t)hd * max_ctx : nullptr;
  const int row0 = act_row(m, vv, b, 0), ld = nkv * hd;
  for (int i = threadIdx.x; i < rows * kp; i += 256) {
    const int r = i / kp, e = i - r * kp;
    qs[i] = (r0 + r < R && e < hd) ? to_f<T>(q[(size_t)(row0 + r0 + r) * nq * hd + (size_t)h * hd + e]) : 0.f;
  }
  const int ra = warp * 2;                      // this warp's rows: ra, ra + 1
  const bool live = ra < rows && r0 + ra < R;
  float* oa = os + ra * hp;
  if (live)
    for (int e = lane; e < 2 * hp; e += 32) oa[e] = 0.f;
  float mx[2] = {-INFINITY, -INFINITY}, sum[2] = {0.f, 0.f};

  const int tc = (P + kt - 1) / kt, ta = (R + kt - 1) / kt;
  for (int t = 0; t < tc + ta; ++t) {
    const bool ctx = t < tc;
    const int j0 = (ctx ? t : t - tc) * kt, n = min(kt, (ctx ? P : R) - j0);
    __syncthreads();                            // the last tile has been read
    // K rows; rows and elements beyond the valid ones are zero
    if (vec) {
      const int q4 = hp / 4;
      for (int i = threadIdx.x; i < kt * q4; i += 256) {
        const int j = i / q4, e = (i - j * q4) * 4;
        float x[4] = {0.f, 0.f, 0.f, 0.f};
        if (j < n) load4<T>((ctx ? kc + (size_t)(j0 + j) * hd : k + (size_t)(row0 + j0 + j) * ld + (size_t)g * hd) + e, x);
        *reinterpret_cast<float4*>(Ks + j * kp + e) = make_float4(x[0], x[1], x[2], x[3]);
      }
    } else {
      for (int i = threadIdx.x; i < kt * hp; i += 256) {
        const int j = i / hp, e = i - j * hp;
        Ks[j * kp + e] = (j < n && e < hd) ? to_f<T>(ctx ? kc[(size_t)(j0 + j) * hd + e]
                                                         : k[(size_t)(row0 + j0 + j) * ld + (size_t)g * hd + e]) : 0.f;
      }
    }
    // V with the keys contiguous; the cache may hold anything beyond ctx_len
    if (ctx && !vec) {
      for (int i = threadIdx.x; i < hd * kt; i += 256) {
        const int e = i / kt, j = i - e * kt;
        Vs[e * vp + j] = j < n ? to_f<T>(vc[(size_t)e * max_ctx + j0 + j]) : 0.f;
      }
    } else if (ctx) {
      for (int i = threadIdx.x; i < hd * (kt / 4); i += 256) {
        const int e = i / (kt / 4), j = (i - e * (kt / 4)) * 4;
        float x[4] = {0.f, 0.f, 0.f, 0.f};
        if (j < n) load4<T>(vc + (size_t)e * max_ctx + j0 + j, x);
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (j + u >= n) x[u] = 0.f;
        *reinterpret_cast<float4*>(Vs + e * vp + j) = make_float4(x[0], x[1], x[2], x[3]);
      }
    } else {
      const int steps = vec ? hd / 4 : hd;
      for (int i = threadIdx.x; i < kt * steps; i += 256) {
        const int e = i / kt, j = i - e * kt;   // lanes along the keys: conflict-free stores
        const T* src = v + (size_t)(row0 + j0 + j) * ld + (size_t)g * hd;
        if (vec) {
          float x[4] = {0.f, 0.f, 0.f, 0.f};
          if (j < n) load4<T>(src + e * 4, x);
#pragma unroll
          for (int u = 0; u < 4; ++u) Vs[(e * 4 + u) * vp + j] = x[u];
        } else {
          Vs[e * vp + j] = j < n ? to_f<T>(src[e]) : 0.f;
        }
      }
    }
    __syncthreads();
    if (!live) continue;
    // scores of the warp's two rows: one key per lane and step
    const float *q0 = qs + ra * kp, *q1 = q0 + kp;
    float *p0 = ps + ra * vp, *p1 = p0 + vp;
    float tm0 = -INFINITY, tm1 = -INFINITY;
    for (int j = lane; j < kt; j += 32) {
      float s0 = -INFINITY, s1 = -INFINITY;
      if (j < n) {
        float a0 = 0.f, a1 = 0.f, b0 = 0.f, b1 = 0.f;
        const float* kr = Ks + j * kp;
        for (int e = 0; e < hp; e += 4) {
          const float4 kv = *reinterpret_cast<const float4*>(kr + e);
          const float4 x = *reinterpret_cast<const float4*>(q0 + e), y = *reinterpret_cast<const float4*>(q1 + e);
          a0 = fmaf(x.x, kv.x, a0); b0 = fmaf(x.y, kv.y, b0); a0 = fmaf(x.z, kv.z, a0); b0 = fmaf(x.w, kv.w, b0);
          a1 = fmaf(y.x, kv.x, a1); b1 = fmaf(y.y, kv.y, b1); a1 = fmaf(y.z, kv.z, a1); b1 = fmaf(y.w, kv.w, b1);
        }
        s0 = (a0 + b0) * scale; s1 = (a1 + b1) * scale;
      }
      p0[j] = s0; p1[j] = s1;
      tm0 = fmaxf(tm0, s0); tm1 = fmaxf(tm1, s1);
    }
    const float n0 = fmaxf(mx[0], warp_max(tm0)), n1 = fmaxf(mx[1], warp_max(tm1));
    const float c0 = expf(mx[0] - n0), c1 = expf(mx[1] - n1);   // 0 on the first tile
    float t0 = 0.f, t1 = 0.f;
    for (int j = lane; j < kt; j += 32) {
      const float e0 = expf(p0[j] - n0), e1 = expf(p1[j] - n1);
      p0[j] = e0; p1[j] = e1;
      t0 += e0; t1 += e1;
    }
    sum[0] = sum[0] * c0 + warp_sum(t0); sum[1] = sum[1] * c1 + warp_sum(t1);
    mx[0] = n0; mx[1] = n1;
    __syncwarp();
    for (int e = lane; e < hd; e += 32) {
      const float* vr = Vs + e * vp;
      float x0 = 0.f, x1 = 0.f, y0 = 0.f, y1 = 0.f;
      for (int j = 0; j < kt; j += 4) {
        const float4 w = *reinterpret_cast<const float4*>(vr + j);
        const float4 x = *reinterpret_cast<const float4*>(p0 + j), y = *reinterpret_cast<const float4*>(p1 + j);
        x0 = fmaf(x.x, w.x, x0); x1 = fmaf(x.y, w.y, x1); x0 = fmaf(x.z, w.z, x0); x1 = fmaf(x.w, w.w, x1);
        y0 = fmaf(y.x, w.x, y0); y1 = fmaf(y.y, w.y, y1); y0 = fmaf(y.z, w.z, y0); y1 = fmaf(y.w, w.w, y1);
      }
      oa[e] = oa[e] * c0 + (x0 + x1);
      oa[hp + e] = oa[hp + e] * c1 + (y0 + y1);
    }
  }
  for (int i = 0; i < 2; ++i) {
    if (!live || r0 + ra + i >= R) break;
    const float inv = 1.f / sum[i];
    T* dst = o + (size_t)(row0 + r0 + ra + i) * nq * hd + (size_t)h * hd;
    for (int e = lane; e < hd; e += 32) dst[e] = from_f<T>(oa[i * hp + e] * inv);
  }
}

// keys per tile, query rows per CTA (two per warp) and shared memory: as many as fit
struct AttnSimtShape { int kt, rows; size_t smem; };
static AttnSimtShape attn_simt_shape(int hd) {
  const size_t hp = (hd + 3) / 4 * 4;
  AttnSimtShape a{64, kAttnSimtRows, 0};
  while (true) {
    a.smem = sizeof(float) * (a.kt * (hp + 4) + (size_t)hd * (a.kt + 4) + a.rows * ((hp + 4) + (a.kt + 4) + hp));
    if (a.smem <= kSimtSmemMax || (a.kt == 4 && a.rows == 2)) return a;
    if (a.kt > 8 || a.rows == 2) a.kt >>= 1; else a.rows >>= 1;
  }
}

// A head_dim whose tiles do not fit in shared memory (above some 3500): a CTA takes one query row of one head and
// keeps it and its output there; K and V are read where they lie, 256 keys at a time.
template <typename T>
__global__ void __launch_bounds__(256) k_attn_simt_wide(
    const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ v,
    const T* __restrict__ k_cache, const T* __restrict__ v_cache, int max_ctx, const SeqMeta m, int nq,
    int nkv, int hd, T* __restrict__ o) {
  extern __shared__ __align__(16) float attn_smem[];
  __shared__ float red[32];
  const int h = blockIdx.y, b = blockIdx.z % m.batch, vv = blockIdx.z / m.batch, g = h / (nq / nkv), r = blockIdx.x;
  const int P = m.ctx_len[b], R = m.last_len[b] + m.win_len[b];
  if (r >= R) return;
  float *qs = attn_smem, *os = qs + hd, *ps = os + hd;   // [hd], [hd], [256]
  const int row0 = act_row(m, vv, b, 0), ld = nkv * hd, tid = threadIdx.x, w = tid >> 5, l = tid & 31;
  const size_t off = (size_t)(row0 + r) * nq * hd + (size_t)h * hd, kvh = (size_t)b * nkv + g;
  for (int e = tid; e < hd; e += 256) { qs[e] = to_f<T>(q[off + e]); os[e] = 0.f; }
  const float scale = rsqrtf((float)hd);
  float mx = -INFINITY, sum = 0.f;
  const int tc = (P + 255) / 256, tiles = tc + (R + 255) / 256;
  for (int t = 0; t < tiles; ++t) {
    const bool ctx = t < tc;
    const int j0 = (ctx ? t : t - tc) * 256, n = min(256, (ctx ? P : R) - j0);
    __syncthreads();                            // the tile before has been read
    float s = -INFINITY;
    if (tid < n) {
      const T* kr = ctx ? k_cache + (kvh * max_ctx + j0 + tid) * hd : k + (size_t)(row0 + j0 + tid) * ld + (size_t)g * hd;
      s = 0.f;
      for (int e = 0; e < hd; ++e) s = fmaf(qs[e], to_f<T>(kr[e]), s);
      s *= scale;
    }
    float top = warp_max(s);
    if (l == 0) red[w] = top;
    __syncthreads();
    for (int i = 0; i < 8; ++i) top = fmaxf(top, red[i]);
    top = fmaxf(top, mx);
    const float corr = expf(mx - top), p = tid < n ? expf(s - top) : 0.f;
    ps[tid] = p;
    sum = sum * corr + block_sum(p, red);       // (its barriers also publish ps)
    mx = top;
    for (int e = tid; e < hd; e += 256) {
      float acc = os[e] * corr;
      if (ctx) {
        const T* vr = v_cache + (kvh * hd + e) * max_ctx + j0;
        for (int j = 0; j < n; ++j) acc = fmaf(ps[j], to_f<T>(vr[j]), acc);
      } else {
        const T* vr = v + (size_t)(row0 + j0) * ld + (size_t)g * hd + e;
        for (int j = 0; j < n; ++j) acc = fmaf(ps[j], to_f<T>(vr[(size_t)j * ld]), acc);
      }
      os[e] = acc;
    }
  }
  const float inv = 1.f / sum;
  for (int e = tid; e < hd; e += 256) o[off + e] = from_f<T>(os[e] * inv);
}
static size_t attn_wide_smem(int hd) { return sizeof(float) * (2 * (size_t)hd + 256); }

template <typename T>
void launch_attn_simt(const T* q, const T* k, const T* v, const T* k_cache, const T* v_cache,
                      int max_ctx, const SeqMeta& m, int nq, int nkv, int hd, T* o,
                      cudaStream_t s) {
  const AttnSimtShape a = attn_simt_shape(hd);
  if (a.smem > kSimtSmemMax) {
    k_attn_simt_wide<T><<<dim3(m.R_cap, nq, m.nv * m.batch), 256, attn_wide_smem(hd), s>>>(q, k, v, k_cache, v_cache, max_ctx, m, nq, nkv, hd, o);
    return;
  }
  auto aligned = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
  const int vec = hd % 4 == 0 && aligned(k_cache) && aligned(v_cache);
  dim3 grid((m.R_cap + a.rows - 1) / a.rows, nq, m.nv * m.batch);
  k_attn_simt<T><<<grid, 256, a.smem, s>>>(q, k, v, k_cache, v_cache, max_ctx, m, nq, nkv, hd, o, a.kt, a.rows, vec);
}

// Opts the kernels of this file in to the shared memory they may ask for, on the current device;
// false when head_dim is too large for the attention kernel's buffers.
template <typename T>
static bool simt_init_t() {
  auto opt = [](auto* f) { return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSimtSmemMax) == cudaSuccess; };
  auto gemm = [&](auto epi) {
    constexpr int E = decltype(epi)::value;
    return opt(k_gemm_simt<T, 1, 1, 8, 128, 3, E>) && opt(k_gemm_simt<T, 4, 2, 1, 32, 3, E>);
  };
  return opt(k_attn_simt<T>) && opt(k_attn_simt_wide<T>) && gemm(std::integral_constant<int, EPI_STORE_F32>{}) &&
         gemm(std::integral_constant<int, EPI_ADD_F32>{}) && gemm(std::integral_constant<int, EPI_SWIGLU>{}) &&
         gemm(std::integral_constant<int, EPI_QKV>{});
}
bool simt_init(bool bf16, int head_dim) {
  // the attributes belong to the functions on a device, not to a context: setting them costs 2 ms,
  // so it is done by the first context of a type on a device (again by a racing one: same values)
  static std::atomic<unsigned long long> done[2];
  int dev = 0;
  cudaGetDevice(&dev);
  const unsigned long long bit = dev < 64 ? 1ull << dev : 0ull;
  bool ok = (done[bf16].load(std::memory_order_acquire) & bit) != 0;
  if (!ok) {
    ok = bf16 ? simt_init_t<__nv_bfloat16>() : simt_init_t<float>();
    if (ok) done[bf16].fetch_or(bit, std::memory_order_release);
    cudaGetLastError();
  }
  return ok && (attn_simt_shape(head_dim).smem <= kSimtSmemMax || attn_wide_smem(head_dim) <= kSimtSmemMax);
}

// ---- per-position signals from full logits (CUDA-core LM head only): one block per window position --
constexpr int kSigThreads = 512;
__global__ void __launch_bounds__(kSigThreads) k_signals(const SimtSignals sg, const SeqMeta m) {
  __shared__ SignalsShared<kSigThreads> sh;
  signals_pos<kSigThreads>(sg, m, blockIdx.x, threadIdx.x, sh, [] { __syncthreads(); });
}

void launch_signals_from_logits(const SimtSignals& sg, const SeqMeta& m, cudaStream_t s) {
  k_signals<<<m.batch * m.W_cap, kSigThreads, 0, s>>>(sg, m);
}

// ---- cross log-probabilities: xlogp[b,i,j] = h_i . W_lm[yhat_j] - lse_i  (Eq. 6 halves) ---------
template <typename T>
__global__ void __launch_bounds__(256) k_xlogp(const T* __restrict__ h,
                                               const T* __restrict__ lm_head,
                                               const int32_t* __restrict__ ws_pred,
                                               const float* __restrict__ ws_lse, int d, int V,
                                               SeqMeta m, int max_window,
                                               float* __restrict__ xlogp) {
  extern __shared__ __align__(16) float wrow[];  // W_lm[yhat_j] as fp32
  pdl_trigger();
  pdl_wait(h, ws_pred, ws_lse);
  const int b = blockIdx.y, j = blockIdx.x;
  const int W = m.win_len[b];
  if (j >= W) return;
  const int tok = ws_pred[b * m.W_cap + j];
  if (tok < 0 || tok >= V) {   // never index the vocabulary matrix with an id outside it
    for (int i = blockIdx.z * (blockDim.x >> 5) + (threadIdx.x >> 5); i < W; i += gridDim.z * (blockDim.x >> 5))
      if ((threadIdx.x & 31) == 0) xlogp[((size_t)b * max_window + i) * max_window + j] = -INFINITY;
    return;
  }
  const T* wr = lm_head + (size_t)tok * d;
  for (int i = threadIdx.x; i < d; i += blockDim.x) wrow[i] = to_f<T>(wr[i]);
  __syncthreads();
  // one window position per warp: blockIdx.z picks the group of positions, so that a step's W * W
  // dot products are spread over W * W / 8 CTAs instead of W (the kernel is bound by the latency
  // of a row load, not by bytes: 37 -> 8 us at W = 64)
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int i = blockIdx.z * nw + warp; i < W; i += gridDim.z * nw) {
    const T* hr = h + (size_t)lm_row(m, 0, b * m.W_cap + i) * d;
    float acc = 0.f;
    // d is a multiple of 4: four elements per lane and step (8- or 16-byte loads), eight steps
    // in flight at a time (the loop is bound by the latency of the h loads otherwise)
    int e = lane * 4;
    for (; e + 7 * 128 < d; e += 8 * 128) {
      float hv[8][4];
#pragma unroll
      for (int u = 0; u < 8; ++u) load4<T>(hr + e + u * 128, hv[u]);
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const float4 wv = *reinterpret_cast<const float4*>(wrow + e + u * 128);
        acc = fmaf(hv[u][0], wv.x, acc); acc = fmaf(hv[u][1], wv.y, acc);
        acc = fmaf(hv[u][2], wv.z, acc); acc = fmaf(hv[u][3], wv.w, acc);
      }
    }
    for (; e < d; e += 128) {
      float hv[4];
      load4<T>(hr + e, hv);
      const float4 wv = *reinterpret_cast<const float4*>(wrow + e);
      acc = fmaf(hv[0], wv.x, acc); acc = fmaf(hv[1], wv.y, acc);
      acc = fmaf(hv[2], wv.z, acc); acc = fmaf(hv[3], wv.w, acc);
    }
    acc = warp_sum(acc);
    if (lane == 0)
      xlogp[((size_t)b * max_window + i) * max_window + j] = acc - ws_lse[b * m.W_cap + i];
  }
}

template <typename T>
void launch_xlogp(const T* h, const T* lm_head, const int32_t* ws_pred, const float* ws_lse, int d,
                  int V, const SeqMeta& m, int max_window, float* xlogp, cudaStream_t s) {
  dim3 grid(m.W_cap, m.batch, (m.W_cap + 7) / 8);
  launch_chained(k_xlogp<T>, grid, 256, d * sizeof(float), s, h, lm_head, ws_pred, ws_lse, d, V, m, max_window, xlogp);
}

// explicit instantiations
#define DC_INST(T)                                                                              \
  template void launch_step_begin<T>(const T*, const int32_t*, const int32_t*, int, int, int, int, \
                                     int, const SeqMeta&, float*, int32_t*, int, float, float*,   \
                                     unsigned int*, int, cudaStream_t);                           \
  template void launch_rmsnorm<T>(float*, const float*, int, size_t, const T*, float, int, int, \
                                  T*, cudaStream_t);                                            \
  template void launch_lm_rows<T>(const float*, const float*, int, size_t, const T*, float, int,  \
                                  const SeqMeta&, int, const LmRowsIo<T>&, T*, cudaStream_t);    \
  template void launch_gemm_simt<T>(const SimtGemm<T>&, int, cudaStream_t);                     \
  template void launch_rope_store<T>(const float*, const SimtGemm<T>&, cudaStream_t);           \
  template void launch_attn_simt<T>(const T*, const T*, const T*, const T*, const T*, int,      \
                                    const SeqMeta&, int, int, int, T*, cudaStream_t);           \
  template void launch_xlogp<T>(const T*, const T*, const int32_t*, const float*, int, int,     \
                                const SeqMeta&, int, float*, cudaStream_t);
DC_INST(float)
DC_INST(__nv_bfloat16)

}  // namespace dc
