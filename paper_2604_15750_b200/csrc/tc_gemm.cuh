// Weight-streaming bf16 GEMM on tcgen05 for the dense layers of the block-step.
//
// out[m, n] = sum_k A[m, k] * W[n, k]        A: activations [M, K], W: weights [N, K]
//
// The step has few activation rows and very many weight rows, so the roles of the MMA operands are
// swapped: a CTA owns 128 weight rows (the MMA "M" side, one TMEM lane per output feature) and a block
// of up to 256 activation rows (the MMA "N" side, one TMEM column per row).  Every weight byte is read
// from HBM exactly once per column block; the activation tile is re-read from L2.
//
// Warp roles (576 threads): warp 0 = TMA producer, warp 1 = TMEM owner + MMA issuer, warps 2..17 =
// epilogue (TMEM -> registers -> global).  Shared memory is a ring of slots, each {NW weight tiles
// 128 x 64, one activation tile BN x 64}, all in the 128-byte swizzled K-major layout that both TMA and
// tcgen05.mma understand.
//
// A CTA works through the units (weight tile, column block, K split) blockIdx.x, + gridDim.x, ...
// The single-matrix GEMMs use one accumulator of up to 256 columns at a time and alternate between two TMEM
// sets: the producer and the MMA issuer run on into the next accumulator and the epilogue of one runs under its
// MMAs.  Gate / up need both sets for one unit; there a CTA's next unit starts when the epilogue has drained them.
//
// The tensor core truncates the running sum at every MMA, so that the error grows with the MMAs of a chain: sums over K =
// 4096 of normal numbers are 4.4e-6 off (relative) in one chain, 2.1e-6 in two, 1.0e-6 in four (of positive ones 1.4e-5,
// 5.3e-6, 2.1e-6); over K = 12288 1.4e-5, 6.7e-6, 3.2e-6.  So the projections back to d go through four accumulators a
// unit, which the epilogue warps add up in registers (0.3 .. 1 us a GEMM against one), and QKV sends even k-steps to the
// one set and odd ones to the other where a CTA has no second unit.
//
// What bounds it: the tensor pipe.  It is busy in 81 .. 87% of an SM's active cycles with 1024 rows of LLaDA-8B and in
// 89 .. 92 with 2560 (O, whose units are short: 65 and 77); the SMs themselves are idle for a fifth to a quarter of a
// launch in last rounds that are not whole, and batches of 2000 rows and more reach the power cap.  Device timestamps with
// 1024 rows showed three other things before: a lane in a branch of its own issued a k-block in 390 ns (the issuing warps now run their loops
// together and elect a lane); the rotation through shared memory by four warps took 27 us a unit against 25 of
// MMAs (shuffles take 3.5: the weight rows arrive in an order that puts the two features of a pair into one warp); gate /
// up stood still for 11 us of every 51 while four warps drained the accumulators (sixteen take 3).  QKV 83 -> 71
// us, gate / up 153 -> 133; the whole prefill 15.1 -> 13.6 ms, eight boundary steps 37.1 -> 33.4.  The four accumulators
// a unit are 0.4% of that prefill, 1.5% of one of 300 rows.
#pragma once
#include "kernels.h"
#include "pdl.cuh"
#include "tc_ptx.cuh"

namespace dc {

enum GemmEpi {
  GEMM_EPI_QKV = 0,      // rotate q/k heads (RoPE), round to bf16, store q, k, v
  GEMM_EPI_PARTIAL = 1,  // fp32 split-K partial sums [split][M][N]
  GEMM_EPI_SWIGLU = 2    // two accumulators (gate, up): bf16 silu(gate) * up
};

struct GemmParams {
  int M;          // valid activation rows
  int N;          // weight rows of one matrix (output features)
  int K;          // reduction length
  int BN;         // activation rows per column block (multiple of 16, <= 256)
  int nsplit;     // split-K factor
  int tiles;      // weight tiles (over all matrices of the call)
  int dual;       // QKV with a unit a worker: two accumulators, even and odd k-steps
  // QKV epilogue
  int nq, nkv;              // tiles [0,nq) are q heads, [nq,nq+nkv) k heads, rest v heads (head_dim 128)
  const float* cos_sin;     // RoPE table [(b, r)][128]
  int rows_per_variant;     // the table is shared by the variants
  const __nv_bfloat16 *bq, *bk, *bv;  // projection biases [nq*hd], [nkv*hd], [nkv*hd], or null
  __nv_bfloat16 *q, *k, *v; // outputs q [M, nq*hd], k [M, nkv*hd], v TRANSPOSED [nkv*hd, ldv]
  int ldv;                  // row pitch of the transposed v (elements, multiple of 8)
  // PARTIAL epilogue
  float* part;              // [nsplit][M_ld][N]
  size_t part_stride;       // elements between splits
  // SWIGLU epilogue
  __nv_bfloat16* act;       // [M, N]
  int32_t* status;          // device status word(s); DC_ERR_TIMEOUT on an expired wait
};

constexpr int kGemmEpiWarps = 16;
constexpr int kGemmParts = kGemmEpiWarps / 4;           // warps per TMEM lane quarter: they share its columns
constexpr int kGemmThreads = 64 + 32 * kGemmEpiWarps;
constexpr int kTileN = 128;  // weight rows per CTA tile
constexpr int kTileK = 64;   // bf16 elements per k-block (one 128-byte swizzle row)
constexpr int kGemmChunks = 256 / (16 * kGemmParts);    // chunks of 16 columns that a warp holds
constexpr int kGemmChains = 4;   // accumulators that a unit of a projection back to d goes through

__host__ __device__ inline int gemm_stage_bytes(int nw, int a_rows) {
  return nw * kTileN * kTileK * 2 + a_rows * kTileK * 2;
}

// Feature of a head (128 wide) in TMEM lane `lane` of quarter q: the weight rows of a q / k / v tile arrive as
// {16 q .. + 15, 64 + 16 q .. + 15} per quarter, so that rotate-half's pair (i, i + 64) lies 16 lanes apart.
__device__ __forceinline__ int head_feature(int quarter, int lane) { return ((lane >> 4) << 6) + 16 * quarter + (lane & 15); }

// The 128 weight rows of head `head` in that order: four boxes of 2 x 16 rows.
template <bool PAIR>
__device__ __forceinline__ void load_head_tile(uint32_t slot, const CUtensorMap* map, uint32_t bar, int kc, int head) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (PAIR) ptx::tma_load_4d_pair_a(slot + q * (32 * kTileK * 2), map, bar, kc, 0, q, 2 * head);
    else ptx::tma_load_4d_a(slot + q * (32 * kTileK * 2), map, bar, kc, 0, q, 2 * head);
  }
}

// PAIR: the launch uses clusters of two CTAs and every MMA is a pair MMA (cta_group::2, M = 256):
// the two CTAs own adjacent weight tiles and each stages only half of the activation block, so a
// k-block is 16 KB of weights plus 16 KB of activations per CTA instead of 16 + 32 - the main
// loops of these GEMMs are close to what an SM takes in from L2.  The even CTA issues the MMAs;
// TMA loads of both CTAs report to its full barrier, tcgen05.commit releases ring slots and
// signals the accumulators in both; the odd CTA's epilogue warps report the drained accumulators
// to the even CTA's barrier.  No load is multicast.
template <int EPI, bool PAIR>
__global__ void __launch_bounds__(kGemmThreads, 1)
k_gemm_tc(const __grid_constant__ CUtensorMap map_w0, const __grid_constant__ CUtensorMap map_w1,
          const __grid_constant__ CUtensorMap map_w2, const __grid_constant__ CUtensorMap map_a,
          const GemmParams p, const int stages) {
  constexpr int NW = (EPI == GEMM_EPI_SWIGLU) ? 2 : 1;
  constexpr int NSETS = 2 / NW;          // accumulator sets that a CTA alternates between
  constexpr int NCH = EPI == GEMM_EPI_PARTIAL ? kGemmChains : 1;
  constexpr int W_BYTES = kTileN * kTileK * 2;
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint64_t bar_full[8], bar_empty[8], acc_full[2], acc_empty[2];
  __shared__ uint32_t tmem_base_s;
  __shared__ int abort_flag, late_flag;
  __shared__ uint32_t fills;             // ring slots that the producer has filled

  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  // Column blocks of one weight tile sit next to each other in the unit order, so that the
  // CTAs that share a weight tile run together and all but one read it from L2.
  const int n_cblk = (p.M + p.BN - 1) / p.BN;
  const uint32_t rank = PAIR ? ptx::cluster_ctarank() : 0u;
  const int cta = PAIR ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;       // worker index: CTA or CTA pair
  const int n_cta = PAIR ? (int)(gridDim.x >> 1) : (int)gridDim.x;
  const int a_rows = PAIR ? p.BN / 2 : p.BN;                             // activation rows this CTA stages
  const int per_split = (PAIR ? p.tiles / 2 : p.tiles) * n_cblk;
  const int n_units = per_split * p.nsplit;
  const int stage_bytes = gemm_stage_bytes(NW, a_rows);
  const int KB = p.K / kTileK;
  constexpr uint32_t tmem_cols = 512u;

  struct Unit { int tile, cblk, split, kb0, nkb; };
  auto unit_of = [&](int u) {
    Unit w;
    w.split = u / per_split;
    const int rem = u - w.split * per_split;
    w.tile = rem / n_cblk;
    w.cblk = rem - w.tile * n_cblk;
    if (PAIR) w.tile = 2 * w.tile + (int)rank;
    w.kb0 = (int)(((long long)w.split * KB) / p.nsplit);
    w.nkb = (int)(((long long)(w.split + 1) * KB) / p.nsplit) - w.kb0;
    return w;
  };

  if (threadIdx.x == 0) {
    abort_flag = 0; late_flag = 0;
    for (int i = 0; i < stages; ++i) { ptx::mbar_init(&bar_full[i], 1); ptx::mbar_init(&bar_empty[i], 1); }
    for (int i = 0; i < 2; ++i) { ptx::mbar_init(&acc_full[i], 1); ptx::mbar_init(&acc_empty[i], (PAIR ? 2 : 1) * kGemmEpiWarps); }
    ptx::fence_barrier_init();
    ptx::prefetch_tmap(&map_w0);
    ptx::prefetch_tmap(&map_a);
    if (NW == 2 || EPI == GEMM_EPI_QKV) ptx::prefetch_tmap(&map_w1);
    if (EPI == GEMM_EPI_QKV) ptx::prefetch_tmap(&map_w2);
  }
  if (warp == 1) {
    ptx::tmem_alloc(&tmem_base_s, tmem_cols, PAIR);
    ptx::tmem_relinquish(PAIR);
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem_base = tmem_base_s;
  pdl_trigger();   // (not before the allocation: pdl.cuh)
  if (PAIR) {
    // both CTAs hold all 512 columns, so the pair MMA's accumulator address names the same columns
    // in both; the partner's barriers are initialised before any load can report to them
    if (threadIdx.x == 0 && tmem_base != 0) abort_flag = 1;
    ptx::cluster_sync();
  }

  const uint32_t full0 = ptx::smem_u32(&bar_full[0]), empty0 = ptx::smem_u32(&bar_empty[0]);
  if (warp == 0) {
    // ---------------- TMA producer ----------------
    // (the whole warp runs the loop and one elected lane issues, as in the MMA issuer)
    const bool el = ptx::elect_one();
    const uint32_t ring0 = ptx::smem_u32(smem);
    const uint32_t full_r0 = (PAIR && rank != 0) ? ptx::mapa_shared(full0, 0) : full0;   // the even CTA's
    // the weight tile(s) of one k-block, and the bytes that the slot's barrier waits for
    auto load_w = [&](const Unit& w, int i, uint32_t s, uint32_t slot) {
      const int kc = (w.kb0 + i) * kTileK;
      if (rank == 0) ptx::mbar_expect_tx_a(full0 + 8u * s, (PAIR ? 2u : 1u) * (uint32_t)stage_bytes);
      const uint32_t bar = full_r0 + 8u * s;
      if (EPI == GEMM_EPI_QKV) {
        const bool is_v = w.tile >= p.nq + p.nkv, is_q = w.tile < p.nq;
        load_head_tile<PAIR>(slot, is_q ? &map_w0 : is_v ? &map_w2 : &map_w1, bar, kc,
                             w.tile - (is_q ? 0 : is_v ? p.nq + p.nkv : p.nq));
      } else if (PAIR) {
        ptx::tma_load_2d_pair_a(slot, &map_w0, bar, kc, w.tile * kTileN);
        if (NW == 2) ptx::tma_load_2d_pair_a(slot + W_BYTES, &map_w1, bar, kc, w.tile * kTileN);
      } else {
        ptx::tma_load_2d_a(slot, &map_w0, bar, kc, w.tile * kTileN);
        if (NW == 2) ptx::tma_load_2d_a(slot + W_BYTES, &map_w1, bar, kc, w.tile * kTileN);
      }
    };
    // The weights of the first slots do not wait for the kernel before this one (nothing in a step writes
    // them, and the step's first launch has waited for all that was in the stream).
    int early = 0;
    if (cta < n_units) {
      const Unit w = unit_of(cta);
      early = w.nkb < stages ? w.nkb : stages;
      for (int i = 0; i < early; ++i)
        if (el) load_w(w, i, (uint32_t)i, ring0 + (uint32_t)(i * stage_bytes));
    }
    pdl_wait();
    uint32_t s = 0, ph = 0, slot = ring0, filled = 0;
    bool ok = true;
    for (int u = cta; u < n_units && ok; u += n_cta) {
      const Unit w = unit_of(u);
      const int arow = w.cblk * p.BN + (int)rank * a_rows;
      for (int i = 0; i < w.nkb; ++i) {
        const bool have_w = early > 0;
        if (have_w) --early;
        else ok = __all_sync(0xffffffffu, ptx::mbar_wait_a(empty0 + 8u * s, ph ^ 1u, &abort_flag));
        if (!ok) break;
        if (el) {
          if (!have_w) load_w(w, i, s, slot);
          const uint32_t bar = full_r0 + 8u * s;
          const int kc = (w.kb0 + i) * kTileK;
          if (PAIR) ptx::tma_load_2d_pair_a(slot + NW * W_BYTES, &map_a, bar, kc, arow);
          else ptx::tma_load_2d_a(slot + NW * W_BYTES, &map_a, bar, kc, arow);
        }
        ++filled;
        if (++s == (uint32_t)stages) { s = 0; ph ^= 1u; slot = ring0; } else slot += (uint32_t)stage_bytes;
      }
    }
    if (el) fills = filled;
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    // The whole warp runs the loop and one elected lane issues: the operands then stay in uniform registers (a
    // k-block of 4 MMAs of 256 columns: 740 clocks in a branch of a single lane, 512 are the tensor core's own).
    if (rank == 0) {
      const bool el = ptx::elect_one();
      const uint32_t idesc = ptx::idesc_bf16(PAIR ? 2 * kTileN : kTileN, p.BN);
      const uint32_t hi = ptx::smem_desc_hi32(), lo0 = ptx::smem_desc_lo(ptx::smem_u32(smem)), step = (uint32_t)stage_bytes >> 4;
      uint32_t s = 0, ph = 0, lo = lo0;
      bool ok = true;
      const uint32_t odd = EPI == GEMM_EPI_QKV && p.dual ? 256u : 0u;   // the odd k-steps' accumulator
      int left = 0;   // k-blocks still to come
      for (int u = cta; u < n_units; u += n_cta) left += unit_of(u).nkb;
      int j = 0;   // accumulators of this CTA so far
      for (int u = cta; u < n_units && ok; u += n_cta) {
        const Unit w = unit_of(u);
        const int nch = min(NCH, w.nkb);
#pragma unroll 1
        for (int ch = 0; ch < nch; ++ch, ++j) {
          const uint32_t set = (uint32_t)(j % NSETS);
          // the epilogue has drained this set (its use before the last one)
          if (j >= NSETS) ok = __all_sync(0xffffffffu, ptx::mbar_wait(&acc_empty[set], (uint32_t)(j / NSETS - 1) & 1u, &abort_flag));
          if (!ok) break;
          ptx::tc_fence_after();
          const uint32_t acc = tmem_base + set * 256u;
          const int i0 = ch * w.nkb / nch, i1 = (ch + 1) * w.nkb / nch;   // its k-blocks
          for (int i = i0; i < i1; ++i) {
            ok = __all_sync(0xffffffffu, ptx::mbar_wait_a(full0 + 8u * s, ph, &abort_flag));
            if (!ok) break;
            const uint32_t more = i > i0 ? 1u : 0u;   // the first MMA of an accumulator overwrites it
            --left;
            if (el) {
              const uint32_t da = lo + (NW * W_BYTES >> 4);
#pragma unroll
              for (int kk = 0; kk < kTileK / 16; ++kk) {
                const uint32_t on = kk > 1 || (kk == 1 && odd == 0) ? 1u : more, to = acc + (kk & 1 ? odd : 0u);
                if (PAIR) {
                  ptx::umma_bf16_pair_lo(to, lo + 2 * kk, da + 2 * kk, hi, idesc, on);
                  if (NW == 2) ptx::umma_bf16_pair_lo(acc + 256u, lo + (W_BYTES >> 4) + 2 * kk, da + 2 * kk, hi, idesc, on);
                } else {
                  ptx::umma_bf16_lo(to, lo + 2 * kk, da + 2 * kk, hi, idesc, on);
                  if (NW == 2) ptx::umma_bf16_lo(acc + 256u, lo + (W_BYTES >> 4) + 2 * kk, da + 2 * kk, hi, idesc, on);
                }
              }
              // Frees the slot in both CTAs, if it is filled once more: an arrival that nobody waits for could come when
              // the partner has left.
              if (left >= stages) {
                if (PAIR) ptx::umma_commit_pair_a(empty0 + 8u * s);
                else ptx::umma_commit_a(empty0 + 8u * s);
              }
            }
            if (++s == (uint32_t)stages) { s = 0; ph ^= 1u; lo = lo0; } else lo += step;
          }
          if (!ok) break;
          if (el) {   // this accumulator is complete (in both CTAs of a pair)
            if (PAIR) ptx::umma_commit_pair(&acc_full[set]);
            else ptx::umma_commit(&acc_full[set]);
          }
        }
      }
    }
  } else {
    // ---------------- epilogue: warps 2..5 and the twelve behind them, TMEM lane quarter = warp % 4 ----------------
    // The four warps of a quarter take chunks of 16 columns (activation rows) in turn.  M is a multiple of 16 (the
    // rows of a sequence are rounded up to that), so a chunk is valid as a whole, and a chunk's rows are consecutive
    // positions of one sequence.
    const int quarter = warp & 3, part = (warp - 2) >> 2;
    const int f = EPI == GEMM_EPI_QKV ? head_feature(quarter, lane) : quarter * 32 + lane;   // feature of the tile in this lane
    const float* cos_sin = p.cos_sin;
    pdl_wait(cos_sin);
    bool ok = true;
    int j = 0;   // accumulators so far
    for (int u = cta; u < n_units && ok; u += n_cta) {
      const Unit w = unit_of(u);
      const int m_base = w.cblk * p.BN, cols = min(p.BN, p.M - m_base);
      auto wait_full = [&]() -> uint32_t {   // this warp's lanes of the next accumulator
        const uint32_t set = (uint32_t)(j % NSETS);
        ok = __all_sync(0xffffffffu, ptx::mbar_wait(&acc_full[set], (uint32_t)(j / NSETS) & 1u, &abort_flag));
        ptx::tc_fence_after();
        return tmem_base + set * 256u + ((uint32_t)(quarter * 32) << 16);
      };
      auto drained = [&]() {
        // the set may be overwritten by the next accumulator but one; the even CTA's MMA issuer waits
        // for the epilogue warps of both CTAs
        ptx::tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          const uint32_t set = (uint32_t)(j % NSETS);
          if (PAIR && rank != 0) ptx::mbar_arrive_remote(ptx::mapa_shared(ptx::smem_u32(&acc_empty[set]), 0));
          else ptx::mbar_arrive(&acc_empty[set]);
        }
        ++j;
      };
      if constexpr (EPI == GEMM_EPI_PARTIAL) {
        float sum[kGemmChunks][16];
#pragma unroll
        for (int k = 0; k < kGemmChunks; ++k)
#pragma unroll
          for (int i = 0; i < 16; ++i) sum[k][i] = 0.f;
#pragma unroll 1
        for (int ch = min(NCH, w.nkb); ch > 0; --ch) {
          const uint32_t t_lane = wait_full();
          if (!ok) break;
#pragma unroll
          for (int k = 0; k < kGemmChunks; ++k)
            if (16 * part + 16 * k * kGemmParts < cols) {
#pragma unroll
              for (int h = 0; h < 16; h += 8) {   // (eight at a time: sixteen more registers are not there)
                float v[8];
                ptx::tmem_ld_32x8(t_lane + 16 * part + 16 * k * kGemmParts + h, v);
                ptx::tmem_ld_wait();
#pragma unroll
                for (int i = 0; i < 8; ++i) sum[k][h + i] += v[i];
              }
            }
          drained();
        }
        if (!ok) break;
#pragma unroll
        for (int k = 0; k < kGemmChunks; ++k) {
          const int c0 = 16 * part + 16 * k * kGemmParts;
          if (c0 >= cols) break;
          float* dst = p.part + (size_t)w.split * p.part_stride + (size_t)(m_base + c0) * p.N + (size_t)(w.tile * kTileN + f);
#pragma unroll
          for (int i = 0; i < 16; ++i, dst += p.N) *dst = sum[k][i];
        }
        continue;
      }
      const bool is_q = w.tile < p.nq, rope = EPI == GEMM_EPI_QKV && w.tile < p.nq + p.nkv;
      float bias_f = 0.f;
      if (EPI == GEMM_EPI_QKV && p.bq != nullptr)
        bias_f = __bfloat162float(is_q ? p.bq[w.tile * 128 + f] : rope ? p.bk[(w.tile - p.nq) * 128 + f]
                                                                       : p.bv[(w.tile - p.nq - p.nkv) * 128 + f]);
      const uint32_t t_lane = wait_full();
      if (!ok) break;
#pragma unroll 1
      for (int c0 = 16 * part; c0 < cols; c0 += 16 * kGemmParts) {
        const int m0 = m_base + c0;
        float v[16], v2[16];   // v2: up, or the odd k-steps' sums
        ptx::tmem_ld_32x16(t_lane + c0, v);
        if (EPI == GEMM_EPI_SWIGLU || p.dual) ptx::tmem_ld_32x16(t_lane + 256u + c0, v2);
        if (EPI == GEMM_EPI_SWIGLU) {
          __nv_bfloat16* dst = p.act + (size_t)m0 * p.N + (size_t)(w.tile * kTileN + f);
          ptx::tmem_ld_wait();
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            // silu(g) = g * (0.5 + 0.5 * tanh(g / 2)): one special-function instruction (as in
            // the fused chain's epilogue; tanh.approx is good to 2^-11, the result goes to bf16)
            float th;
            asm("tanh.approx.f32 %0, %1;" : "=f"(th) : "f"(0.5f * v[i]));
            v[i] = v[i] * fmaf(0.5f, th, 0.5f) * v2[i];
          }
#pragma unroll
          for (int i = 0; i < 16; ++i) dst[(size_t)i * p.N] = __float2bfloat16_rn(v[i]);
          continue;
        }
        // rotate-half: the lane 16 on has the other feature of the pair.  Every row has its own factors from the
        // table, rounded once from fp64: advanced by an angle step from the chunk's first row they were up to 7.7e-7
        // off instead of 3e-8.
        float cv[16], sv[16];
        if (rope) {
          const int mt = m0 >= p.rows_per_variant ? m0 - p.rows_per_variant : m0;   // (prev variant: same table)
          const float* cs = cos_sin + (size_t)mt * 128 + (f & 63);
#pragma unroll
          for (int i = 0; i < 16; ++i) { cv[i] = __ldg(cs + i * 128); sv[i] = __ldg(cs + i * 128 + 64); }
        }
        ptx::tmem_ld_wait();
        if (p.dual)
#pragma unroll
          for (int i = 0; i < 16; ++i) v[i] += v2[i];
        if (!rope) {
          // V is stored transposed (keys contiguous): 16 consecutive keys of feature row f
          __nv_bfloat16* dst = p.v + (size_t)((w.tile - p.nq - p.nkv) * 128 + f) * p.ldv + m0;
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            uint32_t o[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              __nv_bfloat162 pr = __floats2bfloat162_rn(v[8 * h + 2 * e] + bias_f, v[8 * h + 2 * e + 1] + bias_f);
              o[e] = *reinterpret_cast<uint32_t*>(&pr);
            }
            *reinterpret_cast<uint4*>(dst + 8 * h) = make_uint4(o[0], o[1], o[2], o[3]);
          }
        } else {
          const float sg = lane < 16 ? -1.f : 1.f;
          const int ld = (is_q ? p.nq : p.nkv) * 128;
          __nv_bfloat16* dst = (is_q ? p.q + w.tile * 128 : p.k + (w.tile - p.nq) * 128) + (size_t)m0 * ld + f;
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const float y = v[i] + bias_f, other = __shfl_xor_sync(0xffffffffu, y, 16);
            dst[(size_t)i * ld] = __float2bfloat16_rn(fmaf(y, cv[i], sg * other * sv[i]));
          }
        }
      }
      drained();
    }
  }
  ptx::tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && rank == 0 && abort_flag != 0) {
    // given up, whichever role it was (all of them have decided by now): what is still on its way (for the even CTA's
    // barriers, the odd one's loads too) lands before this shared memory goes to another CTA, with a limit of its own
    for (uint32_t n = fills > (uint32_t)stages ? fills - stages : 0; n < fills; ++n)
      ptx::mbar_wait_a(full0 + 8u * (n % stages), (n / stages) & 1u, &late_flag);
  }
  // neither CTA of a pair leaves while the other may still read its shared memory or signal its
  // barriers
  if (PAIR) ptx::cluster_sync();
  if (warp == 1) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem_base, tmem_cols, PAIR);
  }
  if (threadIdx.x == 0 && abort_flag && p.status) atomicExch(p.status, DC_ERR_TIMEOUT);
}

}  // namespace dc
