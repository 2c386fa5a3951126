// Attention of a pass with few active rows (denoising steps above all) on tcgen05, with the operands the
// other way round from tc_attn.cuh: keys on the 128 lanes, query rows on 32 columns.
//
//   S^T [128 keys x 32 rows]  = K Q^T       A = the K tile, B = 32 query rows
//   P^T = exp2(S^T - m0)                    one thread per key: 32 exponentials per tile instead of 128
//   O^T [128 dims x 32 rows] += V^T P^T     A = the V^T tile, B = P (bf16, in shared memory)
//
// Such a pass is bound by the cached keys it streams (64 KB per tile and CTA against a few hundred clocks of
// math).  With 128 rows per tile, most of them padding, the softmax was most of the 2 us that a tile took,
// and one CTA per SM made two waves of it.  Here a CTA takes 32 rows of one (variant, sequence, head), needs
// 128 TMEM columns and - with more CTAs than SMs - a ring of three 32 KB slots, so that two fit on an SM and
// 296 streams run at once; with fewer CTAs than SMs the ring has six slots.  Per layer of LLaDA-8B: eight
// sequences of 900..1200 cached keys, 8..24 rows, 54.5 -> 35.3 us (140 MB: 2.6 -> 4.0 TB/s; the step 6430 ->
// 5871 us); one sequence of 619 keys, 8 rows, 14.3 -> 10.4 us (latency; the step 3676 -> 3539 us).
//
// The reference point m0 of a row is its maximum over the first 32 keys, as in tc_attn.cuh, and no score is
// rescaled.  The sum of a row is at least its largest probability, so a sum above 2^100 tells that some score
// lies too far above m0: then one more pass finds the rows' maxima and a third uses them.
//
// Warp roles (256 threads): warp 0 = TMA producer (Q, then K and V^T tiles in turn through one ring), warp
// 1 = TMEM owner + issuer of S^T, warp 2 = issuer of O^T, warp 3 = clears V^T beyond the valid keys, warps 4..7 =
// softmax and output.
#pragma once
#include "tc_attn.cuh"

namespace dc {

constexpr int kFewThreads = 256;
constexpr int kFewRows = 32;                       // query rows per CTA
constexpr int kFewMaxRows = 64;                    // see few_rows_rule
constexpr int kFewQ = kFewRows * kHd * 2;          // bytes of Q, and of P
constexpr int kFewSlot = 2 * kSub;                 // bytes of a K or V^T tile
constexpr int kFewSlotsMax = 6;                    // (or 3: of tile J, K is in slot 2 J % slots, V^T in the one after)
constexpr float kFewRange = 1.2676506e30f;         // 2^100

// Where this kernel is used (us per layer there -> here):
//  - one variant of up to 64 rows: LLaDA 8 x 1200 keys, 24 rows 58.0 -> 37.7, 48 rows 77.9 -> 68.2, 64 rows 82.3 ->
//    71.4; Dream 8 x 1200, 32 rows 45.0 -> 22.0.  Of 96 rows in many sequences (4 x 512 keys) 44.0 -> 47.4:
//    every further 32 rows stream the keys once more.
//  - any pass that gives every CTA an SM of its own, because the 128-row tiles then leave most SMs idle: one
//    sequence, 96 rows 12.9 -> 10.1, two variants of 48 rows 14.1 -> 12.7.  Beyond that (two variants of 96 rows:
//    192 CTAs) 13.1 -> 13.2, and 38.1 -> 53.9 with 4096 keys.
inline bool few_rows_rule(const SeqMeta& m, int ctas, int n_sm) { return (m.nv == 1 && m.R_cap <= kFewMaxRows) || ctas <= n_sm; }

__host__ __device__ constexpr int few_smem(int slots) { return 2 * kFewQ + slots * kFewSlot + 1024 /*control*/; }

struct FewCtl {
  // Arrivals of K and of V^T tiles have barriers of their own (of tile J: J % 3, with three slots as with six).
  // With three slots the two take turns in a slot, and one barrier per slot, waited on by two issuers, would
  // let the parity of a K tile's phase be taken for that of the phase before the V^T tile in between.
  uint64_t q_full, k_full[3], v_full[3], empty[kFewSlotsMax], s_full[2], s_empty[2], p_full, p_empty;
  uint32_t tmem_base;
  int abort_flag, again_flag, late_flag;
  alignas(16) float m0[kFewRows];      // the rows' reference points (log2 units)
  float part[4][kFewRows];             // per softmax warp: the rows' sums (or maxima) over its keys
  alignas(16) float inv[kFewRows];
};
static_assert(sizeof(FewCtl) <= 1024, "control block");

// Reduces v[row] over the lanes of a warp, all 32 rows at once: lane i returns row i's result.
template <bool MAX>
__device__ __forceinline__ float few_reduce(float (&v)[32], int lane) {
#pragma unroll
  for (int s = 16; s >= 1; s >>= 1) {
    const bool upper = (lane & s) != 0;
#pragma unroll
    for (int i = 0; i < s; ++i) {
      const float send = upper ? v[i] : v[i + s], keep = upper ? v[i + s] : v[i];
      const float got = __shfl_xor_sync(0xffffffffu, send, s);
      v[i] = MAX ? fmaxf(keep, got) : keep + got;
    }
  }
  return v[0];
}

__global__ void __launch_bounds__(kFewThreads, 2)
k_attn_few(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
           const __grid_constant__ CUtensorMap map_vt, const __grid_constant__ CUtensorMap map_kc,
           const __grid_constant__ CUtensorMap map_vc, const AttnParams p, const int slots) {
  extern __shared__ uint8_t smem_few[];
  const int b = blockIdx.z, h = blockIdx.y;
  if ((int)blockIdx.x >= p.units) {
    pdl_trigger();
    pdl_wait();
    const int r0 = ((int)blockIdx.x - p.units) * kBK;
    if (h < p.nkv && r0 < p.m.last_len[b]) attn_export_tile<kFewThreads>(p, b, h, r0);
    return;
  }
  const int P = p.m.ctx_len[b], R = p.m.last_len[b] + p.m.win_len[b];
  const int nqt = p.units / p.m.nv, var = (int)blockIdx.x / nqt;
  const int q0 = ((int)blockIdx.x - var * nqt) * kFewRows, n = min(kFewRows, R - q0);
  if (n <= 0) { pdl_wait(); return; }
  if ((ptx::smem_u32(smem_few) & 1023u) != 0) {   // (it is all the shared memory there is and starts on such a boundary)
    pdl_wait();
    if (threadIdx.x == 0 && p.status) atomicExch(p.status, DC_ERR_UNSUPPORTED);
    return;
  }
  uint8_t *Qs = smem_few, *Ps = smem_few + kFewQ, *ring = smem_few + 2 * kFewQ;
  FewCtl& c = *reinterpret_cast<FewCtl*>(ring + slots * kFewSlot);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = h / (p.nq / p.nkv);
  const int Tc = (P + kBK - 1) / kBK, T = Tc + (R + kBK - 1) / kBK;   // context tiles, then tiles of active keys

  if (threadIdx.x == 0) {
    c.abort_flag = 0; c.again_flag = 0; c.late_flag = 0;
    ptx::mbar_init(&c.q_full, 1);
    for (int i = 0; i < slots; ++i) ptx::mbar_init(&c.empty[i], 1);
    for (int i = 0; i < 3; ++i) { ptx::mbar_init(&c.k_full[i], 1); ptx::mbar_init(&c.v_full[i], 1); }
    for (int i = 0; i < 2; ++i) { ptx::mbar_init(&c.s_full[i], 1); ptx::mbar_init(&c.s_empty[i], 4); }
    ptx::mbar_init(&c.p_full, 5);   // the softmax warps, and warp 3
    ptx::mbar_init(&c.p_empty, 1);
    ptx::fence_barrier_init();
  }
  if (warp == 1) {
    ptx::tmem_alloc(&c.tmem_base, 128);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem_base = c.tmem_base;   // columns: S^T of tile J in buffer J % 2 (0..31, 32..63), O^T 64..95
  pdl_trigger();   // (not before the allocation: pdl.cuh)
  pdl_wait();

  int* abort_flag = &c.abort_flag;
  int loads = 0;   // of the producer thread: Q, then K and V^T tiles
  // Tiles are counted through all passes (J = pass * T + j); the ring holds items 2 J (K) and 2 J + 1 (V^T).
  for (int pass = 0; pass < 3; ++pass) {
    const int J0 = pass * T;
    if (warp == 0) {
      if (lane == 0) {
        // ---------------- TMA producer ----------------
        if (pass == 0) {
          const int row = act_row(p.m, var, b, q0);
          ptx::mbar_expect_tx(&c.q_full, kFewQ);
          ptx::tma_load_2d(Qs, &map_q, &c.q_full, h * kHd, row);
          ptx::tma_load_2d(Qs + kFewQ / 2, &map_q, &c.q_full, h * kHd + 64, row);
          loads = 1;
        }
        int s = (2 * J0) % slots;
        uint32_t ph = (uint32_t)((2 * J0) / slots) & 1u;
        for (int it = 0; it < 2 * T; ++it) {
          const int j = it >> 1;
          if (!ptx::mbar_wait(&c.empty[s], ph ^ 1u, abort_flag)) break;
          uint8_t* dst = ring + (size_t)s * kFewSlot;
          uint64_t* bar = (it & 1) == 0 ? &c.k_full[(J0 + j) % 3] : &c.v_full[(J0 + j) % 3];
          ptx::mbar_expect_tx(bar, kFewSlot);
          if ((it & 1) == 0) {
            if (j < Tc) {
              const int krow = (b * p.nkv + g) * p.max_ctx + j * kBK;
              ptx::tma_load_3d(dst, &map_kc, bar, 0, krow, p.layer);
              ptx::tma_load_3d(dst + kSub, &map_kc, bar, 64, krow, p.layer);
            } else {
              const int row = act_row(p.m, var, b, (j - Tc) * kBK);
              ptx::tma_load_2d(dst, &map_k, bar, g * kHd, row);
              ptx::tma_load_2d(dst + kSub, &map_k, bar, g * kHd + 64, row);
            }
          } else if (j < Tc) {
            const int vrow = (b * p.nkv + g) * kHd;
            ptx::tma_load_3d(dst, &map_vc, bar, j * kBK, vrow, p.layer);
            ptx::tma_load_3d(dst + kSub, &map_vc, bar, j * kBK + 64, vrow, p.layer);
          } else {
            const int col = act_row(p.m, var, b, (j - Tc) * kBK);
            ptx::tma_load_2d(dst, &map_vt, bar, col, g * kHd);
            ptx::tma_load_2d(dst + kSub, &map_vt, bar, col + 64, g * kHd);
          }
          ++loads;
          if (++s == slots) { s = 0; ph ^= 1u; }
        }
      }
    } else if (warp == 1 || warp == 2) {
      // ---------------- issuers of S^T = K Q^T (warp 1) and O^T (+)= V^T P^T (warp 2) ----------------
      const bool pv = warp == 2;
      const uint32_t idesc = ptx::idesc_bf16(128, kFewRows), hi32 = ptx::smem_desc_hi32();
      const uint32_t b_lo = ptx::smem_desc_lo(ptx::smem_u32(pv ? Ps : Qs)), ring_lo = ptx::smem_desc_lo(ptx::smem_u32(ring));
      bool ok = __all_sync(0xffffffffu, pv || ptx::mbar_wait(&c.q_full, 0, abort_flag));
      for (int j = 0; j < T && ok; ++j) {
        const int J = J0 + j, it = 2 * J + (pv ? 1 : 0), s = it % slots;
        if (pv) ok = ptx::mbar_wait(&c.p_full, (uint32_t)J & 1u, abort_flag);
        else if (J >= 2) ok = ptx::mbar_wait(&c.s_empty[J & 1], ((uint32_t)(J - 2) >> 1) & 1u, abort_flag);
        ok = ok && ptx::mbar_wait(pv ? &c.v_full[J % 3] : &c.k_full[J % 3], (uint32_t)(J / 3) & 1u, abort_flag);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        ptx::tc_fence_after();
        if (ptx::elect_one()) {
          const uint32_t d = tmem_base + (pv ? 64u : (uint32_t)(J & 1) * 32u);
          const uint32_t a = ring_lo + (uint32_t)s * (kFewSlot >> 4);
          const int nk = pv ? attn_pv_keys(min(kBK, j < Tc ? P - j * kBK : R - (j - Tc) * kBK)) >> 4 : 8;
#pragma unroll
          for (int kk = 0; kk < 8; ++kk) {
            if (kk >= nk) break;
            const uint32_t k4 = (uint32_t)(kk & 3) * 2u, half = (uint32_t)(kk >> 2);
            ptx::umma_bf16_lo(d, a + half * (kSub >> 4) + k4, b_lo + half * (kFewQ / 2 >> 4) + k4, hi32, idesc,
                              (kk > 0 || (pv && j > 0)) ? 1u : 0u);
          }
          ptx::umma_commit(&c.empty[s]);
          ptx::umma_commit(pv ? &c.p_empty : &c.s_full[J & 1]);
        }
        __syncwarp();
      }
    } else if (warp == 3) {
      // ---------------- V^T columns beyond the valid keys: cleared while the softmax warps make P ----------------
      for (int j = 0; j < T; ++j) {
        const int J = J0 + j, nvalid = min(kBK, j < Tc ? P - j * kBK : R - (j - Tc) * kBK);
        if (nvalid & 15) {
          if (!__all_sync(0xffffffffu, ptx::mbar_wait(&c.v_full[J % 3], (uint32_t)(J / 3) & 1u, abort_flag))) break;
#pragma unroll
          for (int rr = lane; rr < 128; rr += 32) attn_clear_v(ring + (size_t)((2 * J + 1) % slots) * kFewSlot, rr, nvalid);
          ptx::fence_proxy_async_smem();
          __syncwarp();
        }
        if (lane == 0) ptx::mbar_arrive(&c.p_full);
        // (not ahead of the tile: its next arrival belongs to the next phase)
        if (!__all_sync(0xffffffffu, ptx::mbar_wait(&c.p_full, (uint32_t)J & 1u, abort_flag))) break;
      }
    } else if (warp >= 4) {
      // ---------------- softmax: one thread per key of the tile ----------------
      const int quarter = warp & 3, key = quarter * 32 + lane;
      const uint32_t t_lane = tmem_base + ((uint32_t)(quarter * 32) << 16);
      const float scale = p.scale_log2;
      const bool find_max = pass == 1;
      // this key's column of P [32 rows][128 keys]: rows 8 i + e at offset 1024 i from the address of row e
      uint32_t p_addr[8];
#pragma unroll
      for (int e = 0; e < 8; ++e)
        p_addr[e] = ptx::smem_u32(Ps) + (uint32_t)((key >> 6) * (kFewQ / 2) + e * 128 + ((((key & 63) >> 3) ^ e) << 4) + (key & 7) * 2);
      float acc[32];   // the rows' sums over this thread's keys; their maxima in the pass that looks for them
#pragma unroll
      for (int i = 0; i < 32; ++i) acc[i] = find_max ? -INFINITY : 0.f;
      bool ok = true;
      for (int j = 0; j < T; ++j) {
        const int J = J0 + j;
        const int nvalid = min(kBK, j < Tc ? P - j * kBK : R - (j - Tc) * kBK);
        const bool valid = key < nvalid;
        float v[32];
        ok = __all_sync(0xffffffffu, ptx::mbar_wait(&c.s_full[J & 1], ((uint32_t)J >> 1) & 1u, abort_flag));
        if (ok) {
          ptx::tc_fence_after();
          ptx::tmem_ld_32x32(t_lane + (uint32_t)(J & 1) * 32u, v);
          ptx::tmem_ld_wait();
          ptx::tc_fence_before();
          __syncwarp();
          if (lane == 0) ptx::mbar_arrive(&c.s_empty[J & 1]);
        }
        if (J == 0) {   // (every softmax warp comes here, whatever its wait said)
          if (ok && quarter == 0) {   // the first key of the first tile is always valid
            float w[32];
#pragma unroll
            for (int i = 0; i < 32; ++i) w[i] = valid ? v[i] : -INFINITY;
            const float top = few_reduce<true>(w, lane);
            c.m0[lane] = top == -INFINITY ? 0.f : top * scale;
          }
          asm volatile("bar.sync 1, 128;" ::: "memory");
        }
        if (!ok) break;
        // keys beyond the valid length (whatever the cache holds there, NaN included) have probability 0
        if (!find_max) {
#pragma unroll
          for (int i = 0; i < 32; i += 4) {
            const float4 m4 = *reinterpret_cast<const float4*>(&c.m0[i]);
            v[i] = valid ? attn_ex2(fmaf(v[i], scale, -m4.x)) : 0.f;
            v[i + 1] = valid ? attn_ex2(fmaf(v[i + 1], scale, -m4.y)) : 0.f;
            v[i + 2] = valid ? attn_ex2(fmaf(v[i + 2], scale, -m4.z)) : 0.f;
            v[i + 3] = valid ? attn_ex2(fmaf(v[i + 3], scale, -m4.w)) : 0.f;
          }
#pragma unroll
          for (int i = 0; i < 32; ++i) acc[i] += v[i];
        } else {
#pragma unroll
          for (int i = 0; i < 32; ++i) { acc[i] = valid ? fmaxf(acc[i], v[i]) : acc[i]; v[i] = 0.f; }
        }
        // P of the tile before has been read
        if (J > 0) ok = __all_sync(0xffffffffu, ptx::mbar_wait(&c.p_empty, (uint32_t)(J - 1) & 1u, abort_flag));
        if (!ok) break;
#pragma unroll
        for (int i = 0; i < 32; ++i)
          asm volatile("st.shared.b16 [%0], %1;" ::"r"(p_addr[i & 7] + (uint32_t)(i >> 3) * 1024u),
                       "h"(__bfloat16_as_ushort(__float2bfloat16_rn(v[i]))) : "memory");
        ptx::fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(&c.p_full);
      }
      // O^T is complete once the last P has been read
      if (ok) ok = __all_sync(0xffffffffu, ptx::mbar_wait(&c.p_empty, (uint32_t)(J0 + T - 1) & 1u, abort_flag));
      c.part[quarter][lane] = find_max ? few_reduce<true>(acc, lane) : few_reduce<false>(acc, lane);
      asm volatile("bar.sync 1, 128;" ::: "memory");
      if (quarter == 0) {   // lane = row
        if (find_max) {
          const float top = fmaxf(fmaxf(c.part[0][lane], c.part[1][lane]), fmaxf(c.part[2][lane], c.part[3][lane]));
          c.m0[lane] = top == -INFINITY ? 0.f : top * scale;
        } else {
          const float l = (c.part[0][lane] + c.part[1][lane]) + (c.part[2][lane] + c.part[3][lane]);
          c.inv[lane] = 1.f / l;
          const bool far = pass == 0 && lane < n && l > kFewRange;
          if (__any_sync(0xffffffffu, far) && lane == 0) c.again_flag = 1;
        }
      }
    }
    // ---------------- end of the pass: once more, or write the output ----------------
    __syncthreads();
    if (pass < 2 && c.again_flag != 0 && c.abort_flag == 0) continue;
    if (warp >= 4 && c.abort_flag == 0) {
      ptx::tc_fence_after();
      const int quarter = warp & 3;
      float o[32];
      ptx::tmem_ld_32x32(tmem_base + ((uint32_t)(quarter * 32) << 16) + 64u, o);
      ptx::tmem_ld_wait();
      __nv_bfloat16* dst = p.o + (size_t)act_row(p.m, var, b, q0) * p.nq * kHd + (size_t)h * kHd + quarter * 32 + lane;
#pragma unroll
      for (int i = 0; i < 32; ++i)
        if (i < n) dst[(size_t)i * p.nq * kHd] = __float2bfloat16_rn(o[i] * c.inv[i]);
    }
    break;
  }
  if (loads > 0 && c.abort_flag != 0) {
    // given up: what is still on its way lands before another CTA gets this shared memory (with a limit of its own)
    ptx::mbar_wait(&c.q_full, 0, &c.late_flag);
    for (int it = max(0, loads - 7); it < loads - 1; ++it) {   // the last three tiles of each kind
      const int J = it >> 1;
      ptx::mbar_wait((it & 1) == 0 ? &c.k_full[J % 3] : &c.v_full[J % 3], (uint32_t)(J / 3) & 1u, &c.late_flag);
    }
  }
  ptx::tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem_base, 128);
  }
  if (threadIdx.x == 0 && c.abort_flag && p.status) atomicExch(p.status, DC_ERR_TIMEOUT);
}

}  // namespace dc
