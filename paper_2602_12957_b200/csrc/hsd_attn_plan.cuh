// The attention plan of a step: how the q-tiles' KV ranges are cut into the shares of the CTA slots of an attention launch.
#pragma once
#include "hsd_kernels.h"

namespace hsd {

// The unit (share, kv head) that CTA `bx` of a grid of `G` starts with (n: none).  A launch with fewer units than CTAs
// leaves some SMs with one busy CTA (the grid is two CTAs per SM, and CTA b shares its SM with CTA b + G/2 under the usual
// placement); a CTA that has its SM alone walks its blocks faster, so the longest units go to those SMs and the others
// pair a long one with a short one (shares of a one-round plan are sorted longest first).
__device__ __forceinline__ int attn_unit_at(int bx, int n, int G) {
  const int half = G / 2;
  if (n <= half || n > G) return bx;
  const int n_second = n - half;                       // busy CTAs in the second half of the grid
  if (bx < half) return bx >= n_second ? bx - n_second : (half - n_second) + bx;
  return bx - half < n_second ? n - 1 - (bx - half) : n;
}

// ------------------------------------------------------------------------------------------------
// Plan: one CTA, inside the launch that sets the step up.  Work is counted in 64-key blocks.  A kv head has `max_shares` CTA
// slots; every kv head has the same plan, so a launch runs n_shares x n_kv_heads units, unit u = share u / n_kv_heads of
// head u % n_kv_heads.
//
// One round: a q-tile is cut into equal slices of about `chunk` blocks, each a share of its own, as fine as leaves no slot
// with two.  Cutting costs a hand-over (~3 us, five blocks' time), so a q-tile of up to 4/3 min_chunk blocks stays whole, and
// the last slice to finish adds up the others' results (~0.6 us each, about a block's time): n blocks in slices of c take
// c + kSliceCost n / c, which is least at c = sqrt(kSliceCost n).  Measured, steps of the 24-layer decoder in slices of
// 4 / 6 / 8 / 12 / 16 blocks, relative to the best: one q-tile of 32 blocks 1.02 / 1 / 1.03 / 1.05 / 1.13; one of 126 blocks
// 1.20 / 1.09 / 1.05 / 1 / 1.01; two of 75 blocks 1.09 / 1.07 / 1.02 / 1 / 1.04; 16 of 4 to 17 blocks 1 / 1 / 1.01 / 1.01 / 1.06;
// two of 7 blocks cut in half 1.03, whole 1.
// Results are added up three at a time, so a fourth slice costs a round (~1 us): up to kThreeSlices blocks are cut in three
// where four would save two blocks' time at most.  Four slices against three, graph replays of 39 batches of 1 to 12 regions of up
// to 24 blocks (24 layers): 0.98 to 1.02, slower in 19, faster in 8 (one q-tile of 24 blocks 0.983).  Larger counts were not measured.
// Line: where that leaves the longest slice more than kLineGain blocks above the mean, or above kLineGain (more q-tiles than slots, or
// q-tiles a little longer than the mean, which only halves would shorten), the q-tiles' ranges are laid end to end, each
// with kTileCost blocks added for what an item costs beside its blocks (Q, first product, output), and the line is cut into
// equal shares; a cut that would leave a piece of fewer than kMinPiece blocks moves to the q-tile's edge.
// Measured, step times with equal shares of the line always against one round always: 2,048 rows over 16,384 (33
// q-tiles of 272 blocks on 37 slots) 0.94; 16 regions (25 q-tiles of 4 to 17 blocks) 1.03; 512 rows over 7,936 1.025.
// no_cut (contexts with a fixed summation order): q-tiles are never cut, cuts of the line move to the nearer edge.
constexpr float kSliceCost = 1.4f;
constexpr int kTileCost = 3, kMinPiece = 2, kLineGain = 8, kPlanTiles = 512, kThreeSlices = 24;
template <int THREADS>
__device__ void make_attn_plan(const RowMeta& rm, const AttnPlan& pl, const KvView& kv, const AttnPlanRule& rule, int n_seqs,
                               int n_tiles, int tokens_per_tile) {
  const int max_shares = rule.max_shares, min_chunk = rule.min_chunk, whole = 4 * min_chunk / 3;
  const bool no_cut = rule.no_cut;
  // one round: creation order of the items; line: cuts (q-tile, block) and how many of them lie inside q-tiles so far
  __shared__ int s_ct[kAttnMaxShares + 1], s_co[kAttnMaxShares + 1], s_rank[kAttnMaxShares + 1];
  __shared__ int s_tile_blocks[kPlanTiles];             // lengths of the first q-tiles (the others: from the metadata)
  __shared__ int s_warp[THREADS / 32], s_longest, s_blocks, s_count, s_slice;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) s_longest = s_blocks = 0;
  for (int s = tid; s < n_seqs; s += THREADS)
    for (int t = rm.seq_tile0[s]; t < rm.seq_tile0[s + 1]; ++t) pl.tile_seq[t] = s;
  __syncthreads();
  auto count_blocks = [&](int t) -> int {              // 64-key blocks q-tile t can see
    const int s = pl.tile_seq[t];
    return (rm.seq_len[s] + min(rm.seq_n[s], (t - rm.seq_tile0[s] + 1) * tokens_per_tile) + 63) >> 6;
  };
  auto blocks_of = [&](int t) -> int { return t < kPlanTiles ? s_tile_blocks[t] : count_blocks(t); };
  auto tile_item = [&](int t, int& tok0) -> int4 {
    const int s = pl.tile_seq[t];
    tok0 = (t - rm.seq_tile0[s]) * tokens_per_tile;
    return make_int4(rm.seq_q0[s] + tok0, rm.seq_len[s] + tok0, min(tokens_per_tile, rm.seq_n[s] - tok0), rm.seq_slot[s]);
  };
  // exclusive sum over the CTA, in thread order; `all` = the total (every thread calls it the same number of times)
  auto scan = [&](int v, int& all) -> int {
    int incl = v;
    for (int o = 1; o < 32; o <<= 1) {
      const int x = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += x;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    int before = 0;
    all = 0;
    for (int w = 0; w < THREADS / 32; ++w) {
      if (w < warp) before += s_warp[w];
      all += s_warp[w];
    }
    __syncthreads();
    return before + incl - v;
  };
  // lengths, and where every q-tile begins on the line
  int total = 0;
  for (int t0 = 0; t0 < n_tiles; t0 += THREADS) {
    const int t = t0 + tid;
    const int n = t < n_tiles ? count_blocks(t) : 0;
    if (t < n_tiles && t < kPlanTiles) s_tile_blocks[t] = n;
    int all;
    const int pos = scan(t < n_tiles ? n + kTileCost : 0, all);
    if (t < n_tiles) {
      pl.tile_pos[t] = total + pos;
      atomicMax(&s_longest, n);
      atomicAdd(&s_blocks, n);
    }
    total += all;
  }
  __syncthreads();
  const int longest = s_longest, mean = (s_blocks + max_shares - 1) / max_shares;
  const int shortest = rule.fine ? min_chunk : max(min_chunk, (int)ceilf(sqrtf(kSliceCost * (float)longest)));
  // one round: the slice length is grown until the items fit the slots
  int chunk = max(shortest, mean);
  auto slices_of = [&](int n) -> int {
    if (n <= whole) return 1;
    const int ns = (n + chunk - 1) / chunk;
    return ns == 4 && n <= kThreeSlices && !rule.fine ? 3 : ns;
  };
  bool line = n_tiles > max_shares;
  if (no_cut) {
    chunk = longest;
  } else if (!line) {
    for (;;) {                                            // every thread runs the same iterations
      if (tid == 0) s_count = s_slice = 0;
      __syncthreads();
      for (int t = tid; t < n_tiles; t += THREADS) {
        const int n = blocks_of(t), ns = slices_of(n);
        atomicAdd(&s_count, ns);
        atomicMax(&s_slice, (n + ns - 1) / ns);
      }
      __syncthreads();
      const int count = s_count;
      __syncthreads();
      if (count <= max_shares || chunk >= longest) break;
      chunk += max(1, chunk >> 5);
    }
    line = s_slice > max(max(mean, shortest), kLineGain) + kLineGain;
  }
  int P;
  if (!line) {
    P = 0;
    for (int t0 = 0; t0 < n_tiles; t0 += THREADS) {
      const int t = t0 + tid;
      const int n = t < n_tiles ? blocks_of(t) : 0;
      const int ns = t < n_tiles ? slices_of(n) : 0;
      int all;
      const int at = P + scan(ns, all);
      for (int k = 0; k < ns; ++k) {                     // q-tile, slice (| slices << 16), length of item at + k
        s_ct[at + k] = t;
        s_co[at + k] = k | (ns << 16);
        s_rank[at + k] = n / ns + (k < n % ns ? 1 : 0);
      }
      P += all;
    }
    __syncthreads();
    for (int i = tid; i < P; i += THREADS) {         // longest first (rank sort, ties by creation order)
      const int len = s_rank[i], t = s_ct[i], k = s_co[i] & 0xffff, ns = s_co[i] >> 16;
      int rank = 0;
      for (int j = 0; j < P; ++j) rank += (s_rank[j] > len) || (s_rank[j] == len && j < i);
      const int n = blocks_of(t), from = k * (n / ns) + min(k, n % ns);
      int tok0;
      pl.items[2 * rank] = tile_item(t, tok0);
      pl.items[2 * rank + 1] = make_int4(from | ((from + len) << 16), k | (ns << 8) | (tok0 << 16), i - k, 0);
      pl.share_start[rank] = rank;
    }
    if (tid == 0) pl.share_start[P] = P;
  } else {
    P = max(1, min(min(max_shares, pl.slots / 2), total / shortest));
    for (int k = tid; k <= P; k += THREADS) {
      int t = n_tiles, off = 0;
      if (k < P) {
        const int b = (int)((long long)k * total / P);
        int lo = 0, hi = n_tiles;                          // last q-tile that begins at or before b
        while (hi - lo > 1) {
          const int mid = (lo + hi) >> 1;
          if (pl.tile_pos[mid] <= b) lo = mid; else hi = mid;
        }
        t = lo;
        const int n = blocks_of(t);
        off = b - pl.tile_pos[t] - kTileCost;
        if (off < kMinPiece || (no_cut && 2 * off < n)) {
          off = 0;
        } else if (no_cut || n - off < kMinPiece) {
          ++t;
          off = 0;
        }
      }
      s_ct[k] = t;
      s_co[k] = off;
    }
    __syncthreads();
    if (warp == 0) {
      int sum = 0;
      for (int k0 = 0; k0 <= P; k0 += 32) {
        const int k = k0 + lane;
        const unsigned in = __ballot_sync(0xffffffffu, k <= P && s_co[min(k, P)] > 0);
        if (k <= P) s_rank[k] = sum + __popc(in & (0xffffffffu >> (31 - lane)));
        sum += __popc(in);
      }
    }
    __syncthreads();
    // a share begins with item (its q-tile + the cuts inside q-tiles up to it); a q-tile's slices follow one another
    for (int k = tid; k <= P; k += THREADS) pl.share_start[k] = s_ct[k] + s_rank[k];
    for (int t = tid; t < n_tiles; t += THREADS) {
      int lo = 0, hi = P;                                  // first cut inside q-tile t or beyond it (cut P lies beyond all)
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (s_ct[mid] > t || (s_ct[mid] == t && s_co[mid] > 0)) hi = mid; else lo = mid + 1;
      }
      const int k0 = lo;
      int ns = 1;
      while (k0 + ns - 1 <= P && s_ct[k0 + ns - 1] == t) ++ns;
      int tok0;
      const int4 ia = tile_item(t, tok0);
      const int n = blocks_of(t), first = t + s_rank[k0] - (s_co[k0] > 0 ? 1 : 0);
      int from = 0;
      for (int k = 0; k < ns; ++k) {
        const int to = k + 1 < ns ? s_co[k0 + k] : n;
        pl.items[2 * (first + k)] = ia;
        pl.items[2 * (first + k) + 1] = make_int4(from | (to << 16), k | (ns << 8) | (tok0 << 16), 2 * (k0 - 1) + 1, 1);
        from = to;
      }
    }
  }
  if (tid == 0) *pl.n_shares = P;
  // slice-arrival counters: zero at the start of a step, reset by the combiner
  for (int i = tid; i < (line ? 2 : 1) * P * pl.n_kv_heads * pl.quarters; i += THREADS) pl.counters[i] = 0;
  // what every CTA of the attention grid starts with, in one record: its first item and the physical blocks of that
  // item's first two KV blocks, so that a CTA's first loads do not wait for a chain of dependent reads (item -> block table)
  __syncthreads();
  for (int b = tid; b < pl.grid; b += THREADS) {
    const int share = attn_unit_at(b, P * pl.n_kv_heads, pl.grid) / pl.n_kv_heads;
    const int i0 = share < P ? pl.share_start[share] : 0, count = share < P ? pl.share_start[share + 1] - i0 : 0;
    if (count == 0) {
      pl.first[3 * b + 2] = make_int4(0, 0, 0, 0);
      continue;
    }
    const int4 ia = pl.items[2 * i0], ib = pl.items[2 * i0 + 1];
    const int kt_lo = ib.x & 0xffff, kt_hi = ib.x >> 16;
    int phys0 = 0, phys1 = 0;
    if (kt_hi > kt_lo && ia.w >= 0 && ia.w < kv.n_slots && kt_hi <= kv.max_blocks) {
      const int* bt = kv.block_table + (size_t)ia.w * kv.max_blocks;
      phys0 = bt[kt_lo];
      phys1 = bt[kt_lo + 1 < kt_hi ? kt_lo + 1 : kt_lo];
    }
    pl.first[3 * b] = ia;
    pl.first[3 * b + 1] = ib;
    pl.first[3 * b + 2] = make_int4(i0, count, phys0, phys1);
  }
}

}  // namespace hsd
