// Decision kernels: the DepGA-Block boundary scan (Section 4.2, cumulative form Section 4.4)
// and CAP-Decoding (Section 4.3, Algorithm 1).  One warp per sequence, more where that is too long a chain
// (k_boundary_wide, select_long).
//
// Every floating-point step that decides an integer is written with explicit round-to-nearest
// intrinsics (no contraction into FMA) and a fixed operation order, so the decisions are a
// function of the input bits alone; running sums use 2^40 fixed point, which is order-free.
#include <math.h>
#include <string.h>

#include <type_traits>

#include "decisions.cuh"
#include "pdl.cuh"

namespace dc {

const SeqMeta kNoLengths{};            // (the lengths are in device memory)
constexpr int kWideBoundary = 4096;   // sequences that k_boundary_wide takes
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

// Windows above 128 on four warps a sequence: eight positions a lane are a chain of their own, and the general
// smoothing more so (radius 1 / 3, W 256, us a call: 1 sequence 13.7 / 15.6 on one warp, 11.8 / 11.7 here; 4096 sequences
// 21.8 / 27.5 and 21.1 / 21.8)
__global__ void __launch_bounds__(128) k_boundary_wide(const float* influence, const float* entropy, const __grid_constant__ SeqMeta m,
                                                       DevLens dl, Hyper hp, BoundaryIo io) {
  __shared__ float sI[33 * (kMaxW / 32)], sH[33 * (kMaxW / 32)];
  __shared__ BoundaryTeam<4> team;
  pdl_trigger();
  pdl_wait();
  boundary_seq<kMaxW / 128, 4>(influence, entropy, blockIdx.x, m, dl, hp, io, sI, sH, &team);
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
  if (max_window > 128 && batch <= kWideBoundary) {
    launch_chained(k_boundary_wide, batch, 128, 0, s, influence, entropy, m, dl, hp, io);
    return;
  }
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
  boundary(influence, entropy, ld, batch, kNoLengths, dl, hp, max_window, score, cum_i, cum_s, block_len, s);
}

// ---- CAP-Decoding ------------------------------------------------------------------------------
// Algorithm 1 with the conflicts evaluated where they decide something: only a member of S removes
// candidates, so D_ij is read for i in S and j still alive - a row and a column of xlogp per selected
// position, never the matrix of the whole pool (Eq. 6: conflict iff xlogp[i,j] + xlogp[j,i] > gamma).
// Position 32 q + lane belongs to the lane; a set of candidates is the array of their sort keys, 0 where
// a position is not in it.  The kernel is bound by instruction issue and by the latency of those
// rows and columns, so the code is kept to few instructions and to the registers of 40 warps per SM.
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
  // 64 positions per round of loads, shorter blocks skip the rest; 128 where one position has 256 to look at (1.0 us
  // instead of 1.6)
  constexpr int G = NA == 1 && NQ >= 8 ? 4 : 2;
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

// Greedy pass over the candidates in confidence order: take a position, drop what conflicts with it.  With
// long_from<NQ>() candidates left after eight positions (few conflict) it gives up: `pending` is set, and select_long
// makes the sequence's selection.  Where the two take as long, candidates at the start of a pass without conflicts:
// 8192 x 128 some 70 (56: 98 us here, 135 there; 80: 243 and 202), one sequence of 128 some 40 (56: 30 and 22), of 256
// about 30.  Up to 64 positions this loop is the faster one to the end (24 us).
template <int NQ>
__device__ __forceinline__ unsigned long_from(int seqs) { return seqs > 1 ? 64u : 32u; }
template <int NQ>
__device__ __forceinline__ unsigned greedy(const float* __restrict__ xb, unsigned ld, int L, unsigned (&key)[NQ], float gamma, int seqs,
                                           bool& pending) {
  unsigned sel = 0u;   // bit q: position 32 q + lane
  for (int picks = 1;; ++picks) {
    const int a[1] = {first_of<NQ>(key)};
    if (a[0] < 0) return sel;
    const bool mine = (int)(threadIdx.x & 31) == (a[0] & 31);
#pragma unroll
    for (int q = 0; q < NQ; ++q)
      if (mine && q == (a[0] >> 5)) { key[q] = 0u; sel |= 1u << q; }
    drop_conflicts<NQ, 1>(xb, ld, L, a, key, gamma);
    if (NQ >= 4 && picks == 8) {
      unsigned left = 0u;
#pragma unroll
      for (int q = 0; q < NQ; ++q) left += key[q] != 0u ? 1u : 0u;
      if (__reduce_add_sync(kAll, left) >= long_from<NQ>(seqs)) { pending = true; return sel; }
    }
  }
}

constexpr int kSelectCtas = 5 * 148;   // CTAs of eight warps that the machine holds at once

// the inputs of a selection, and where it goes
struct SelectArgs {
  const float* conf;
  const int32_t* win_ids;
  const float* xlogp;
  const int32_t* block_len;
  int batch, mask_id, max_window;
  uint8_t* sel_mask;
  int32_t *sel_idx, *sel_count;
  int seqs;   // sequences of a CTA (one per warp; the other warps are there for select_long)
  int vec;    // xlogp starts on a 16-byte boundary
  DevLens dl;
  Hyper hp;
};

// lengths of sequence b: window, block
__device__ __forceinline__ void select_lengths(const SelectArgs& p, const PrevLen& win, const SelectCommit& cm, int b, int& W, int& blk) {
  W = len_of(p.dl.win_len, win.n, b);
  const int kept = cm.win_ids != nullptr ? cm.keep.n[b] : -1;   // the length of a block that a generation is in the middle of
  blk = kept >= 0 ? kept : p.block_len[b];
}

// mask, ascending index list and count of sequence b, by one warp.  sel: bit q is position 32 q + lane; masked: the
// positions of the block that hold a mask.
template <int NQ>
__device__ __forceinline__ void select_store(const SelectArgs& p, const SelectCommit& cm, int b, int W, int blk, unsigned sel, unsigned masked) {
  const int lane = threadIdx.x & 31;
  const size_t o = (size_t)b * p.max_window;
  int total = 0;
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const int k = 32 * q + lane;
    const bool on = (sel >> q) & 1u;
    const unsigned word = __ballot_sync(kAll, on);
    if (p.sel_mask && k < W) p.sel_mask[o + k] = on ? 1 : 0;
    if (p.sel_idx && on) p.sel_idx[o + total + __popc(word & ((1u << lane) - 1u))] = k;
    total += __popc(word);
  }
  if (lane == 0 && p.sel_count) p.sel_count[b] = total;
  if (cm.win_ids == nullptr) return;
  // Eq. (2) and what the host loop of a generation reads, straight into its pinned buffer
  int left = 0;
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const int k = 32 * q + lane;
    left += __popc(__ballot_sync(kAll, ((masked & ~sel) >> q) & 1u));
    if (k < W) {
      int id = p.win_ids[o + k];
      if ((sel >> q) & 1u) { id = cm.pred_id[o + k]; cm.win_ids[o + k] = id; }
      cm.host_ids[o + k] = id;
    }
  }
  if (lane == 0) { cm.host_blk[b] = blk; cm.host_left[b] = left; cm.host_status[b] = cm.status[b]; }
}

__device__ __forceinline__ unsigned select_key(const SelectArgs& p, size_t at) {   // 0: not masked
  const float c = p.conf[at];
  const int id = p.win_ids[at];
  const unsigned key = c == c ? order_key(c) : 1u;
  return id != p.mask_id ? 0u : key;
}
__device__ __forceinline__ void select_bars(const Hyper& hp, unsigned& low, unsigned& high) {
  auto bar = [](float tau) { return tau == tau ? order_key(tau) : kAll; };         // (nothing reaches a NaN)
  low = bar(hp.tau_low); high = max(low, bar(hp.tau_high));
}

// The selection of a sequence with a long greedy pass, by all warps of a CTA: the conflicts of the whole pool as a bit
// matrix, whose loads use whole sectors and do not wait for one another, then a walk over the pool in confidence
// order that only reads bits.  (A position a round is bound by the column of each, 32 sectors a load of which 4
// bytes are used: 14 clocks a sector, with four positions a round as with one.  Without a conflict, one sequence of 256
// positions: 441 us -> 57, of 128: 63 -> 31; 8192 of 128: 907 -> 318.)
template <int NQ>
struct LongPass {
  unsigned key[32 * NQ];         // sort keys of the block's masked positions
  unsigned confl[32 * NQ][NQ];
  unsigned cand[NQ];             // the pool
  unsigned char order[32 * NQ];  // the pool by rank
};
// Conflicts, a tile at a time: 32 positions j, a lane each, and 8 positions i: eight rows at the lanes' columns, and
// eight columns of the lanes' rows, a sector each
template <int NQ>
__device__ __forceinline__ void long_matrix(const float* __restrict__ xb, unsigned ld, LongPass<NQ>& sm, int* next, float gamma, int vec) {
  const int lane = threadIdx.x & 31;
#pragma unroll 1
  while (true) {
    int tile = 0;
    if (lane == 0) tile = atomicAdd(next, 1);
    tile = __shfl_sync(kAll, tile, 0);
    // tile 4 k + s: sub-group s of block pair k = (ib, jb), ib <= jb (the matrix is symmetric)
    int k = tile >> 2, jb = 0;
    while (k > jb) { k -= jb + 1; ++jb; }
    if (jb >= NQ) return;
    const int ib = k, i0 = 32 * ib + 8 * (tile & 3), j = 32 * jb + lane;
    const unsigned ci = (sm.cand[ib] >> (i0 & 31)) & 0xffu, cj = sm.cand[jb];
    unsigned words = 0u, bits = 0u;
    if (ci != 0u && cj != 0u) {
      const bool on = (cj >> lane) & 1u;
      float row[8], col[8];
      const float* cp = xb + (size_t)j * ld + i0;
      if (vec && on) {
        const float4 c0 = *reinterpret_cast<const float4*>(cp), c1 = *reinterpret_cast<const float4*>(cp + 4);
        col[0] = c0.x; col[1] = c0.y; col[2] = c0.z; col[3] = c0.w; col[4] = c1.x; col[5] = c1.y; col[6] = c1.z; col[7] = c1.w;
      } else {
#pragma unroll
        for (int t = 0; t < 8; ++t) col[t] = on ? cp[t] : 0.f;
      }
#pragma unroll
      for (int t = 0; t < 8; ++t) row[t] = on ? xb[(unsigned)(i0 + t) * ld + j] : 0.f;
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        const bool c = on && ((ci >> t) & 1u) && __fadd_rn(row[t], col[t]) > gamma;
        const unsigned word = __ballot_sync(kAll, c);
        if (lane == t) words = word;
        bits |= (c ? 1u : 0u) << t;
      }
    }
    if (lane < 8) sm.confl[i0 + lane][jb] = words;   // (i itself may be among them: it is taken before)
    if (ib != jb) reinterpret_cast<unsigned char*>(&sm.confl[j][ib])[tile & 3] = (unsigned char)bits;
  }
}

// Sequences first + i, i a bit of `todo`, one after the other, by the warps of `team`: a warp walks over the matrix of
// one while the others make that of the next.  It starts from the inputs again: nothing of the sequences that end
// without it has to be kept for it.
template <int NQ>
__device__ __forceinline__ void select_long(const SelectArgs& p, const PrevLen& win, const SelectCommit& cm, int first, unsigned todo,
                                            unsigned team, LongPass<NQ> (&sm)[2], int& next) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int me = __popc(team & ((1u << w) - 1u)), n_team = __popc(team);
  auto sync = [&]() { asm volatile("barrier.cta.sync 2, %0;" ::"r"(32 * n_team) : "memory"); };
  unsigned k_low, k_high;
  select_bars(p.hp, k_low, k_high);
  int before = -1;
#pragma unroll 1
  for (int turn = 0;; ++turn) {
    LongPass<NQ>& lp = sm[turn & 1];
    const int cur = todo != 0u ? first + __ffs(todo) - 1 : -1;
    todo &= todo - 1u;
    if (cur >= 0) {
      int W, blk;
      select_lengths(p, win, cm, cur, W, blk);
      const int L = min(max(blk, 0), W);
#pragma unroll 1
      for (int q = me; q < NQ; q += n_team) {
        const int k = 32 * q + lane;
        const unsigned key = k < L ? select_key(p, (size_t)cur * p.max_window + k) : 0u;
        lp.key[k] = key;
        const unsigned word = __ballot_sync(kAll, key != 0u && key >= k_low);
        if (lane == 0) lp.cand[q] = word;
      }
      if (me == 0 && lane == 0) next = 0;
      sync();
#pragma unroll 1
      for (int q = me; q < NQ; q += n_team) {   // rank: higher keys, and as high ones in front
        const int k = 32 * q + lane;
        const unsigned key = lp.key[k];
        int r = 0;
#pragma unroll 2
        for (int s = 0; s < 32 * NQ; s += 4) {
          const uint4 o = *reinterpret_cast<const uint4*>(&lp.key[s]);
          r += (o.x + (s < k ? 1u : 0u) > key ? 1 : 0) + (o.y + (s + 1 < k ? 1u : 0u) > key ? 1 : 0) +
               (o.z + (s + 2 < k ? 1u : 0u) > key ? 1 : 0) + (o.w + (s + 3 < k ? 1u : 0u) > key ? 1 : 0);
        }
        if ((lp.cand[q] >> lane) & 1u) lp.order[r] = (unsigned char)k;
      }
    }
    if (before >= 0 && me == turn % n_team) {
      // Algorithm 1 in one walk: the positions of phase 1 come first, and as printed all of them are taken.  Lane q holds
      // word q of the sets.
      const LongPass<NQ>& lw = sm[(turn & 1) ^ 1];
      const bool literal = p.hp.cap_mode != DC_CAP_STRICT;
      unsigned alive = lane < NQ ? lw.cand[lane] : 0u, taken = 0u, masked = 0u;
      const int n = (int)__reduce_add_sync(kAll, (unsigned)__popc(alive));
#pragma unroll 1
      for (int t = 0; t < n; ++t) {
        const int i = lw.order[t], q = i >> 5;
        const unsigned c = lane < NQ ? lw.confl[i][lane] : 0u, bit = 1u << (i & 31);
        const bool always = literal && lw.key[i] >= k_high;
        if ((__shfl_sync(kAll, alive, q) & bit) == 0u && !always) continue;
        alive &= ~c;
        if (lane == q) { taken |= bit; alive &= ~bit; }
      }
      unsigned sel = 0u;
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        sel |= ((__shfl_sync(kAll, taken, q) >> lane) & 1u) << q;
        masked |= (lw.key[32 * q + lane] != 0u ? 1u : 0u) << q;
      }
      int W, blk;
      select_lengths(p, win, cm, before, W, blk);
      select_store<NQ>(p, cm, before, W, blk, sel, masked);
    }
    if (cur < 0) return;
    long_matrix<NQ>(p.xlogp + (size_t)cur * p.max_window * p.max_window, p.max_window, lp, &next, p.hp.gamma, p.vec);
    sync();
    before = cur;
  }
}

template <int NQ>
__global__ void __launch_bounds__(32 * kSeqWarps, 5) k_select(const __grid_constant__ SelectArgs p, const __grid_constant__ PrevLen win,
                                                              const __grid_constant__ SelectCommit cm) {
  constexpr int NA = 4;
  constexpr bool kCoop = NQ >= 4;             // (shorter windows have no long passes)
  __shared__ __align__(16) int members[kSeqWarps][32 * NQ + NA];
  __shared__ __align__(16) LongPass<kCoop ? NQ : 1> lp[2];
  __shared__ int lp_next, lp_pending[kSeqWarps];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int b = blockIdx.x * p.seqs + w;
  bool pending = false;
  pdl_wait();
  if (w < p.seqs && b < p.batch) {
    int W, blk;
    select_lengths(p, win, cm, b, W, blk);
    const int L = min(max(blk, 0), W);
    const size_t o = (size_t)b * p.max_window;
    const float* xb = p.xlogp + o * p.max_window;
    unsigned key[NQ];                         // M^t ∩ B^t
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      const int k = 32 * q + lane;
      key[q] = k < L ? select_key(p, o + k) : 0u;
    }
    unsigned k_low, k_high;
    select_bars(p.hp, k_low, k_high);
    unsigned cand[NQ];
    unsigned sel = 0u;
    if (p.hp.cap_mode == DC_CAP_STRICT) {     // phase 1, greedily with conflict checks
#pragma unroll
      for (int q = 0; q < NQ; ++q) cand[q] = key[q] >= k_high ? key[q] : 0u;
      sel = greedy<NQ>(xb, p.max_window, L, cand, p.hp.gamma, p.seqs, pending);
    } else {                                  // phase 1 as printed: every c_i >= tau_high enters S
#pragma unroll
      for (int q = 0; q < NQ; ++q) sel |= (key[q] >= k_high ? 1u : 0u) << q;
    }
    if (!pending) {
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
      unsigned left = 0u;
#pragma unroll
      for (int q = 0; q < NQ; ++q) left |= cand[q];
      if (!__any_sync(kAll, left != 0u)) n = 0;
      for (int t = 0; t < n; t += NA) {
        const int4 g = *reinterpret_cast<const int4*>(&members[w][t]);
        const int a[NA] = {g.x, g.y, g.z, g.w};
        drop_conflicts<NQ, NA>(xb, p.max_window, L, a, cand, p.hp.gamma);
      }
      // phase 2: greedy completion in descending confidence
      sel |= greedy<NQ>(xb, p.max_window, L, cand, p.hp.gamma, p.seqs, pending);
    }
    if (!pending) {
      // fallback: the most confident masked position of the block
      if (!__any_sync(kAll, sel != 0u)) {
        const int a = first_of<NQ>(key);
        if (a >= 0 && lane == (a & 31)) sel = 1u << (a >> 5);
      }
      unsigned masked = 0u;
#pragma unroll
      for (int q = 0; q < NQ; ++q) masked |= (key[q] != 0u ? 1u : 0u) << q;
      select_store<NQ>(p, cm, b, W, blk, sel, masked);
    }
  }
  if constexpr (kCoop) {
    // Warps that are done only arrive and leave (waiting for the slowest one cost 3 of 47 us at 8192 x 128); those of
    // an open sequence and those without one end the open ones.
    if (lane == 0) lp_pending[w] = pending ? 1 : 0;
    __syncwarp();
    if (!pending && w < p.seqs) {
      asm volatile("barrier.cta.arrive 1, %0;" ::"r"(blockDim.x) : "memory");
      return;
    }
    asm volatile("barrier.cta.sync 1, %0;" ::"r"(blockDim.x) : "memory");
    const unsigned todo = __ballot_sync(kAll, lane < p.seqs && lp_pending[lane & (kSeqWarps - 1)] != 0);
    const unsigned idle = (1u << (blockDim.x >> 5)) - (1u << p.seqs);
    if (todo != 0u) select_long<NQ>(p, win, cm, blockIdx.x * p.seqs, todo, todo | idle, lp, lp_next);
  }
}

static void select(const float* conf, const int32_t* win_ids, const float* xlogp, const int32_t* block_len, int batch,
                   const SeqMeta& m, const DevLens& dl, const Hyper& hp, int mask_id, int max_window,
                   uint8_t* sel_mask, int32_t* sel_idx, int32_t* sel_count, cudaStream_t s,
                   const SelectCommit& cm = SelectCommit{}) {
  PrevLen win;
  memcpy(win.n, m.win_len, sizeof(win.n));
  SelectArgs p{conf, win_ids, xlogp, block_len, batch, mask_id, max_window, sel_mask, sel_idx, sel_count, 0,
               (reinterpret_cast<uintptr_t>(xlogp) & 15) == 0 ? 1 : 0, dl, hp};
  decide_launch(batch, max_window, [&](auto nq, dim3 grid, int threads) {
    constexpr int NQ = decltype(nq)::value;
    p.seqs = threads / 32;
    if (NQ >= 4) {
      // Whole CTAs, which end long passes together: the machine is filled before a CTA gets a second sequence.  Calls that
      // would put more than six into one have CTAs of four warps, whose slots are free sooner (boundary and
      // selection of 6000 x 128: 35.9 us against 38.4; below, the larger CTAs are the better spread: 1500 x 128 16.3
      // against 18.0, 4000 x 128 27.8 and 27.8).
      const int warps = NQ == 4 && batch > 6 * kSelectCtas ? kSeqWarps / 2 : kSeqWarps, ctas = kSelectCtas * kSeqWarps / warps;
      p.seqs = (batch + ctas - 1) / ctas;
      if (p.seqs > warps) p.seqs = warps;
      threads = 32 * warps;
      grid = dim3((batch + p.seqs - 1) / p.seqs);
    }
    launch_chained(k_select<NQ>, grid, threads, 0, s, p, win, cm);
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
  select(conf, win_ids, xlogp, block_len, batch, kNoLengths, dl, hp, mask_id, max_window, sel_mask, sel_idx, sel_count, s);
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
