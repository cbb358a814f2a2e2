// Varlen multi-query-token causal attention over the paged KV cache, tcgen05 / TMEM / TMA (sm_100a).
//
// A draft token attends to every committed row of its sequence and, causally, to the draft rows before it
// (the chain case of the paper's tree-ancestry mask, Sec. 3.2 / Fig. 2(c)).
//
// Work item = (q-tile, kv slice, kv head).  A q-tile is 128 MMA rows: 128/group consecutive tokens of one
// sequence x the `group` query heads that share the kv head (GQA packing, so K/V blocks are read once per
// group).  A q-tile's KV range is run whole or cut into slices so that a launch has one share of work per CTA slot,
// whatever the mix of context lengths (one page chunk over a long context, or many short regions); the plan is made
// once per step on the device (make_attn_plan) and reused by every layer.  Slices leave
// (unnormalised O, exponent reference, sum) partials in the workspace and the last slice to finish combines them in
// slice order, so the result does not depend on which CTA ran what.
//
// The KV range is walked in paged blocks of 64 keys [64 keys][head_dim] per kv head, fetched by TMA through the block
// table; K is the K-major B operand of S = Q K^T (128 x 64 x head_dim), V the MN-major B operand of O += P V (128 x
// head_dim x 64).  Persistent CTAs, two per SM, walk their shares.  Warp roles:
//   warp 0      TMA producer: Q, the K ring and the V ring
//   warp 1      MMA issuer + TMEM owner
//   warps 2..5  softmax: warp w works on TMEM lane quarter w mod 4 (the hardware's rule), one thread per q row
// Per block: S (TMEM, 64 fp32 columns) -> softmax in registers -> P (bf16) over the same columns, the A operand of the
// second product, so P never passes through shared memory -> O += P V accumulated in tensor memory.  NBUF score
// buffers rotate: while the softmax warps work on block t, S(t + 1) .. S(t + NBUF - 1) are formed already, and the
// buffer of block t is taken by S(t + NBUF) once the product that reads P(t) has completed.  Nothing in the softmax
// warps' loop waits for a product of the same block.
//
// What bounds it: the exp unit, 16 results per clock and SM, i.e. 512 cycles for the 128 x 64 scores of a block, and
// the softmax warps' own dependent chain around it.  One thread owns a row, so a row's threads have nothing to agree
// on, and the exponent reference does not wait for a maximum: it is the maximum of the first 64 keys the row saw, later
// exponentials start as soon as their scores are in registers, and the row sum, which is needed anyway, shows whether a
// score has outgrown the reference (P and the sums are scale-free in bf16 / fp32 as long as they stay in range).  Where
// a sum of 64 exceeds kRescaleSum the 64 are taken again under a new reference and the accumulator row is rescaled.
// Measured, one launch of a 2,048-row chunk over 16,384 committed rows: 245 us with 16 / 8 heads of 64, 145 us with 8
// heads of 128; with two threads a row that agree on a maximum first, on 128-key tiles with one score buffer, a fifth longer.
// Every wait is a bounded mbarrier wait, so one that gives up takes the whole CTA to the common exit.
#include "hsd_attn_plan.cuh"
#include "hsd_kernels.h"

namespace hsd {

constexpr int kSoftmaxWarps = 4;
constexpr int kAttnThreads = 32 * (2 + kSoftmaxWarps);
constexpr int SUB_BYTES = 128 * 128;               // one K-major operand sub-tile of Q: 128 rows x 64 dims
constexpr int KV_BLOCK_BYTES = 64 * 128;           // one paged block of K or of V for one kv head, 64 dims of it
constexpr int ATTN_BAR_BYTES = 256;
constexpr float kRescaleSum = 1099511627776.f;     // 2^40: a row's 64 exponentials that sum to more ask for a new reference
// Head dimension HD = 64 or 128.  An operand tile is HD / 64 sub-tiles of 64 dims each (a 128-byte-swizzled row is 64
// bf16): Q [sub][128 rows][64], a K or V stage [sub][64 keys][64].  The accumulator has HD columns and NBUF score
// buffers of 64 share the 256 columns with it, so two CTAs fit the 512 columns of an SM at either head size.
// No alignment slack: two CTAs of this size plus the per-CTA reserve share an SM, so the kernel relies on the 1024-byte
// alignment it declares for its dynamic shared memory (the swizzled tiles need it) and checks it.
template <int HD>
struct AttnCfg {
  static constexpr int NSUB = HD / 64;
  static constexpr int Q_BYTES = NSUB * SUB_BYTES;
  static constexpr int KV_BYTES = NSUB * KV_BLOCK_BYTES;           // one stage of a ring: 64 keys
  static constexpr int STAGES = HD == 64 ? 4 : 2;                  // per ring
  static constexpr int SMEM = Q_BYTES + 2 * STAGES * KV_BYTES + ATTN_BAR_BYTES;
  static constexpr int TMEM_COLS = 256;
  static constexpr int COL_O = TMEM_COLS - HD, NBUF = COL_O / 64;  // score buffers at columns 64 b
};

struct AttnParams {
  AttnPlan plan;
  const int* block_table;
  int max_blocks, n_blocks, Hq, Hkv, group, layer;
  bf16* out;            // [T, Hq*HD]
  float* split_ws;      // partials of sliced items: [slot][kv head][quarter][32 (2 + HD)], see slice_slot
  const uint4* anc;     // [T] ancestry masks of candidate-tree rows, or nullptr: plain causal order within the call
  int* status;
};

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// packed pairs: one instruction for two fp32 operations
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  float2 d;
  asm("{\n\t.reg .b64 ra, rb, rc, rd;\n\t"
      "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\tmov.b64 rc, {%6, %7};\n\t"
      "fma.rn.f32x2 rd, ra, rb, rc;\n\tmov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return d;
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  float2 d;
  asm("{\n\t.reg .b64 ra, rb, rd;\n\t"
      "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
      "add.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float y;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(y) : "f"(a), "f"(b), "f"(c));
  return y;
}
// Where the partials of a sliced q-tile's slices lie.  One-round plans: every item has a slot of its own, `z` names slice
// 0's.  Line plans: z = 2 k0 + 1 with k0 the share whose last item is slice 0; slice k > 0 is the first item of share
// k0 + k, so two slots per share keep all slices apart.  Either way z is unique to the q-tile (its arrival counter).
__device__ __forceinline__ int slice_slot(int z, int slice, int line) { return !line ? z + slice : slice == 0 ? z : z - 1 + 2 * slice; }

// ------------------------------------------------------------------------------------------------
template <int HD>
__global__ void __launch_bounds__(kAttnThreads, 2)
attn_sm100_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                  const __grid_constant__ CUtensorMap tmV, AttnParams p) {
  using C = AttnCfg<HD>;
  constexpr int NSUB = C::NSUB, STAGES = C::STAGES, NBUF = C::NBUF;
  extern __shared__ __align__(1024) uint8_t smem[];
  uint8_t* sQ = smem;
  uint8_t* sK = sQ + C::Q_BYTES;                       // ring stage s: sK + s * C::KV_BYTES, per sub-tile 64 keys
  uint8_t* sV = sK + STAGES * C::KV_BYTES;
  uint64_t* bars = reinterpret_cast<uint64_t*>(sV + STAGES * C::KV_BYTES);
  uint64_t* q_full = bars;                 // Q tile landed                       (one phase per item)
  uint64_t* q_empty = bars + 1;            // every S MMA of the item has read Q   (one phase per item)
  uint64_t* k_full = bars + 2;             // [stage]
  uint64_t* k_empty = k_full + STAGES;     // [stage] S of the block has been formed
  uint64_t* v_full = k_empty + STAGES;
  uint64_t* v_empty = v_full + STAGES;     // [stage] O += P V of the block has completed
  uint64_t* s_full = v_empty + STAGES;     // [buffer] S(t) is in tensor memory
  uint64_t* p_full = s_full + NBUF;        // [buffer] P(t) is in tensor memory (and the accumulator rescaled, if it had to be)
  uint64_t* o_full = p_full + NBUF;        // [buffer] O += P(t) V(t) has completed.  (One barrier for all blocks would not do:
                                           // a wait for block t passes on the parity of t - 2 where t - 1 is still running.)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(o_full + NBUF);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (smem_u32(smem) & 1023u) {            // uniform over the CTA: nothing has been set up yet
    if (threadIdx.x == 0) dev_fail(p.status, DEV_WAIT_TIMEOUT, 499);
    return;
  }
  // The plan's record of this CTA's first item (the item and the physical blocks of its first keys) for the two warps
  // that start the pipeline: read together with the status word and the share count, ahead of the CTA's own set-up, so that
  // the first TMA loads do not wait for a chain of dependent reads (status -> count -> item -> block table).
  // (Read after the set-up, with the first item's Q behind its K and V, a CTA that cannot start early forms its first
  // scores 0.9 us later.)
  // All of it, like the block table and the K/V rows committed before this step, was written before the kernel that
  // precedes this one in the step: that kernel waited for ITS predecessor before it let this one start, so these reads
  // need no wait of their own, and the first K/V blocks load while the predecessor (which writes q and this step's own
  // K/V rows) is still running.  They go to L2, where completed kernels have left it: a line that an earlier launch put into
  // this SM's L1 may be a former step's.
  int4 rec_a = make_int4(0, 0, 0, 0), rec_b = rec_a, rec_c = rec_a;
  if (warp < 2) {
    const int4* rec = p.plan.first + 3 * (size_t)blockIdx.x;
    rec_a = __ldcg(rec);
    rec_b = __ldcg(rec + 1);
    rec_c = __ldcg(rec + 2);
  }
  const int status_now = __ldcg(p.status), n_shares_now = __ldcg(p.plan.n_shares);
  if (threadIdx.x == 32) {
    tma_prefetch_desc(&tmK);
    tma_prefetch_desc(&tmV);
    tma_prefetch_desc(&tmQ);
  }
  if (threadIdx.x == 0) {
    mbar_init(q_full, 1);
    mbar_init(q_empty, 1);
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(k_full + s, 1);
      mbar_init(k_empty + s, 1);
      mbar_init(v_full + s, 1);
      mbar_init(v_empty + s, 1);
    }
    for (int b = 0; b < NBUF; ++b) {
      mbar_init(s_full + b, 1);
      mbar_init(p_full + b, kSoftmaxWarps);
      mbar_init(o_full + b, 1);
    }
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, C::TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  const int n_units = status_now ? 0 : n_shares_now * p.Hkv;
  const int G = (int)gridDim.x, u0 = attn_unit_at((int)blockIdx.x, n_units, G);

  // Block counter t (all 64-key blocks of all items of this CTA): ring stage = t % STAGES, score buffer = t % NBUF, and
  // every barrier's parity follows from how often t has used it; n counts items (Q hand-over barriers).
  //
  // The producer and the MMA warp run their loops as whole warps and elect one lane for the instructions that one thread
  // issues: with warp-uniform control flow descriptors and coordinates live in uniform registers, where those
  // instructions want them (run by lane 0 alone, an MMA took ~90 cycles to issue; elected, ~25).
  if (warp == 0) {
    uint32_t t = 0;                                      // the K blocks of t + 1 go out before the V block of t
    int n = 0;
    auto load = [&](const CUtensorMap* tm, uint8_t* ring, uint64_t* full, uint64_t* empty, uint32_t at, int phys, int kvh) -> bool {
      const int st = at % STAGES;
      if (!mbar_wait(empty + st, ((at / STAGES) & 1) ^ 1u, abort_flag, p.status, 401)) return false;
      const int row = (((p.layer * p.n_blocks) + phys) * p.Hkv + kvh) * 64;
      if (elect_one()) {
        mbar_expect_tx(full + st, C::KV_BYTES);
#pragma unroll
        for (int h = 0; h < NSUB; ++h) tma_load_2d(ring + st * C::KV_BYTES + h * KV_BLOCK_BYTES, tm, full + st, 64 * h, row);
      }
      __syncwarp();
      return true;
    };
    bool waited = false;                                 // for the kernel before this one
    for (int u = u0; u < n_units; u += G) {
     const int kvh = u % p.Hkv;
     const int i0 = u == u0 ? rec_c.x : p.plan.share_start[u / p.Hkv];
     const int i1 = u == u0 ? rec_c.x + rec_c.y : p.plan.share_start[u / p.Hkv + 1];
     for (int i = i0; i < i1; ++i) {
      const bool recorded = u == u0 && i == i0;
      const int4 ia = recorded ? rec_a : p.plan.items[2 * i], ib = recorded ? rec_b : p.plan.items[2 * i + 1];
      const int kt_lo = ib.x & 0xffff, kt_hi = ib.x >> 16;
      const int* bt = p.block_table + (size_t)ia.w * p.max_blocks;
      auto phys_of = [&](int kt) -> int { return recorded && kt < kt_lo + 2 ? (kt == kt_lo ? rec_c.z : rec_c.w) : __ldcg(bt + kt); };
      int early = kt_lo;                                 // K and V of [kt_lo, early) are on their way
      if (recorded) {
        // blocks that hold committed rows only, as many as the rings take, ahead of the grid dependency
        const int committed = min(kt_hi, (ia.y - (ib.y >> 16)) >> 6);
        for (; early < committed && early - kt_lo < STAGES; ++early) {
          const int phys = phys_of(early);
          if (!load(&tmK, sK, k_full, k_empty, t + (early - kt_lo), phys, kvh)) goto done;
          if (!load(&tmV, sV, v_full, v_empty, t + (early - kt_lo), phys, kvh)) goto done;
        }
      }
      if (!waited) {
        pdl_wait();
        waited = true;
      }
      if (!recorded) {                                   // (the first item's Q: the MMA warp)
        if (!mbar_wait(q_empty, (n & 1) ^ 1u, abort_flag, p.status, 400)) goto done;
        if (elect_one()) {
          mbar_expect_tx(q_full, C::Q_BYTES);
#pragma unroll
          for (int h = 0; h < NSUB; ++h) tma_load_3d(sQ + h * SUB_BYTES, &tmQ, q_full, 64 * h, kvh * p.group, ia.x);
        }
        __syncwarp();
      }
      int phys_v = early < kt_hi ? phys_of(early) : 0;
      if (early < kt_hi && !load(&tmK, sK, k_full, k_empty, t + (early - kt_lo), phys_v, kvh)) goto done;
      for (int kt = early; kt < kt_hi; ++kt) {
        int phys_k = 0;
        if (kt + 1 < kt_hi) {
          phys_k = phys_of(kt + 1);
          if (!load(&tmK, sK, k_full, k_empty, t + (kt + 1 - kt_lo), phys_k, kvh)) goto done;
        }
        if (!load(&tmV, sV, v_full, v_empty, t + (kt - kt_lo), phys_v, kvh)) goto done;
        phys_v = phys_k;
      }
      t += kt_hi - kt_lo;
      ++n;
     }
    }
  } else if (warp == 1) {
    pdl_wait();
    pdl_launch_dependents();
    if (u0 < n_units && rec_c.y > 0 && elect_one()) {    // Q of the first item, beside the producer's K and V
      mbar_expect_tx(q_full, C::Q_BYTES);
#pragma unroll
      for (int h = 0; h < NSUB; ++h) tma_load_3d(sQ + h * SUB_BYTES, &tmQ, q_full, 64 * h, (u0 % p.Hkv) * p.group, rec_a.x);
    }
    __syncwarp();
    constexpr uint32_t idesc_s = umma_idesc_bf16(64);
    constexpr uint32_t idesc_pv = umma_idesc_bf16(64, true);
    const uint64_t q_desc = umma_desc_sw128(smem_u32(sQ)), k_desc = umma_desc_sw128(smem_u32(sK)),
                   v_desc = umma_desc_sw128(smem_u32(sV));     // a byte offset adds a sixteenth of itself
    uint32_t t = 0;
    int n = 0;
    for (int u = u0; u < n_units; u += G) {
     const int i0 = u == u0 ? rec_c.x : p.plan.share_start[u / p.Hkv];
     const int i1 = u == u0 ? rec_c.x + rec_c.y : p.plan.share_start[u / p.Hkv + 1];
     for (int i = i0; i < i1; ++i) {
      const int4 ib = u == u0 && i == i0 ? rec_b : p.plan.items[2 * i + 1];
      const uint32_t t_end = t + (ib.x >> 16) - (ib.x & 0xffff);
      // S(ti) = Q K(ti)^T: four K = 16 steps over every 64 dims, N = 64 keys, into the buffer P(ti - NBUF) has left
      auto issue_s = [&](uint32_t ti) -> bool {
        const int st = ti % STAGES;
        if (!mbar_wait(k_full + st, (ti / STAGES) & 1, abort_flag, p.status, 410)) return false;
        tc_fence_after();
        const uint64_t kd = k_desc + st * (C::KV_BYTES / 16);
        const uint32_t buf = ti % NBUF;
        if (elect_one()) {
#pragma unroll
          for (int h = 0; h < NSUB; ++h)
#pragma unroll
            for (int k = 0; k < 4; ++k)
              umma_bf16(tmem_base + 64 * buf, q_desc + (h * SUB_BYTES + k * 32) / 16, kd + (h * KV_BLOCK_BYTES + k * 32) / 16,
                        idesc_s, (h | k) != 0);
          umma_commit(s_full + buf);
          umma_commit(k_empty + st);              // K is free once S has been formed
          if (ti + 1 == t_end) umma_commit(q_empty);   // last S MMA of the item: Q is free once it completes
        }
        __syncwarp();
        return true;
      };
      // the last product of the item before has completed: every buffer is free
      if (t > 0 && !mbar_wait(o_full + (t - 1) % NBUF, ((t - 1) / NBUF) & 1, abort_flag, p.status, 411)) goto done;
      if (!mbar_wait(q_full, n & 1, abort_flag, p.status, 412)) goto done;
      for (uint32_t ti = t; ti < t_end && ti < t + NBUF; ++ti)
        if (!issue_s(ti)) goto done;
      for (bool first = true; t < t_end; ++t, first = false) {
        const int st = t % STAGES;
        const uint32_t buf = t % NBUF;
        if (!mbar_wait(v_full + st, (t / STAGES) & 1, abort_flag, p.status, 415)) goto done;
        // P(t) is written, and whatever had to be done to the accumulator before this product is done
        if (!mbar_wait(p_full + buf, (t / NBUF) & 1, abort_flag, p.status, 413)) goto done;
        tc_fence_after();
        const uint64_t vd = v_desc + st * (C::KV_BYTES / 16);
        if (elect_one()) {
#pragma unroll
          for (int h = 0; h < NSUB; ++h)   // 64 output dims per product
#pragma unroll
            for (int k = 0; k < 4; ++k)
              // 16 keys per step: 8 columns of P in tensor memory; V [key][dim] is MN-major, a step of 16 keys is 16
              // rows of 128 bytes; the first product of an item overwrites the accumulator
              umma_bf16_ta(tmem_base + C::COL_O + 64 * h, tmem_base + 64 * buf + k * 8, vd + (h * KV_BLOCK_BYTES + k * 2048) / 16,
                           idesc_pv, (!first || k != 0) ? 1u : 0u);
          umma_commit(o_full + buf);
          umma_commit(v_empty + st);
        }
        __syncwarp();
        if (t + NBUF < t_end) {
          if (!mbar_wait(o_full + buf, (t / NBUF) & 1, abort_flag, p.status, 416)) goto done;
          if (!issue_s(t + NBUF)) goto done;
        }
      }
      ++n;
     }
    }
    // every stage-release arrival must land before the CTA's shared memory can be handed on
    if (t > 0 && !mbar_wait(o_full + (t - 1) % NBUF, ((t - 1) / NBUF) & 1, abort_flag, p.status, 414)) goto done;
    if (t > 0 && !mbar_wait(v_empty + (t - 1) % STAGES, ((t - 1) / STAGES) & 1, abort_flag, p.status, 417)) goto done;
  } else {
    const int quarter = warp & 3;                      // TMEM lane quarter a warp may touch = warp id mod 4
    const int row = quarter * 32 + lane;               // q row of the tile = TMEM lane
    const int tok = row / p.group;
    const uint32_t t_lane = tmem_base + (uint32_t(quarter * 32) << 16);
    const uint32_t t_o = t_lane + C::COL_O;
    const float sc = (HD == 64 ? 0.125f : 0.08838834764831845f) * 1.4426950408889634f;     // 1/sqrt(HD) * log2(e)
    uint32_t t = 0;
    pdl_wait();
    for (int u = u0; u < n_units; u += G) {
     const int kvh = u % p.Hkv;
     const int i0 = p.plan.share_start[u / p.Hkv], i1 = p.plan.share_start[u / p.Hkv + 1];
     for (int i = i0; i < i1; ++i) {
      const int4 ia = p.plan.items[2 * i], ib = p.plan.items[2 * i + 1];
      const int q_row0 = ia.x, pos0 = ia.y, n_tok = ia.z;
      const int kt_lo = ib.x & 0xffff, kt_hi = ib.x >> 16;
      const int split = ib.y & 0xff, n_split = (ib.y >> 8) & 0xff;
      const int pos_row = pos0 + tok;
      const bool row_ok = tok < n_tok;
      // candidate trees (Sec. 3.2, Fig. 2(c)): a row sees the committed context and, of the rows of this call, only
      // itself and its ancestors.  len0 = committed length; the mask's bit i stands for cache row len0 + i.
      const int len0 = pos0 - (ib.y >> 16);
      uint4 am = make_uint4(0u, 0u, 0u, 0u);
      if (p.anc && row_ok) am = p.anc[q_row0 + tok];
      // warp-uniform: some row of this warp is a real token.  A ragged last q-tile leaves whole warps without one;
      // they keep step with the barriers but skip the loads, the exps and the P rows (which only feed their own,
      // never stored, output rows)
      const bool warp_ok = (quarter * 32) / p.group < n_tok;
      // exponent reference (log2 units, scaled; a row that is no token asks for none); sum of the row's P
      float m_ref = row_ok ? -INFINITY : 0.f, l = 0.f;
      // visibility of the 32 keys from `key0` on for this thread's row, as a bit mask
      auto visible = [&](int key0) -> uint32_t {
        if (p.anc) {
          auto word = [&](int i) -> uint32_t {
            return i < 0 ? 0xffffffffu : i == 0 ? am.x : i == 1 ? am.y : i == 2 ? am.z : i == 3 ? am.w : 0u;
          };
          const int pos = key0 - len0;
          if (pos <= -32) return 0xffffffffu;
          if (pos >= 128) return 0u;
          const int wi = pos >> 5;                      // floor, also for negative positions
          return __funnelshift_r(word(wi), word(wi + 1), pos & 31);
        }
        const int nvis = pos_row - key0 + 1;            // keys key0 .. pos_row are visible
        return nvis >= 32 ? 0xffffffffu : (nvis <= 0 ? 0u : ((1u << nvis) - 1u));
      };
      const int first_masked = p.anc ? len0 : pos0 + 1;  // keys below it are visible to every row of the q-tile

      for (int kt = kt_lo; kt < kt_hi; ++kt, ++t) {
        const uint32_t buf = t % NBUF;
        bool ok = mbar_wait(s_full + buf, (t / NBUF) & 1, abort_flag, p.status, 420);
        if (!__all_sync(0xffffffffu, ok)) goto done;
        tc_fence_after();
        if (warp_ok) {
          const uint32_t t_s = t_lane + 64 * buf;
          uint32_t a[32], b[32], pk[32];
          tmem_ld32(t_s, a);
          tmem_ld32(t_s + 32, b);
          tmem_ld_wait(a);
          tmem_ld_wait(b);
          if (kt * 64 + 63 >= first_masked) {            // (warp-uniform)
            const uint32_t va = visible(kt * 64), vb = visible(kt * 64 + 32);
#pragma unroll
            for (int e = 0; e < 32; ++e) {
              if (!((va >> e) & 1u)) a[e] = 0xff800000u;               // -inf
              if (!((vb >> e) & 1u)) b[e] = 0xff800000u;
            }
          }
          bool retake = m_ref == -INFINITY;              // no reference yet: it is the maximum of these 64 scores
          float sum;
          for (;;) {
            if (__any_sync(0xffffffffu, retake)) {
              float mx = -INFINITY, mx_b = -INFINITY;    // two chains
#pragma unroll
              for (int e = 0; e < 32; e += 2) {
                mx = max3(mx, __uint_as_float(a[e]), __uint_as_float(b[e]));
                mx_b = max3(mx_b, __uint_as_float(a[e + 1]), __uint_as_float(b[e + 1]));
              }
              mx = fmaxf(mx, mx_b) * sc;
              // Rows that ask for it, and only those (a row's result does not depend on its neighbours), take the new
              // reference and rescale what they have accumulated, once the product before has completed.
              float alpha = 1.f;
              if (retake) {
                if (m_ref != -INFINITY) alpha = ex2(m_ref - mx);
                m_ref = mx;
                l *= alpha;
              }
              if (__any_sync(0xffffffffu, alpha != 1.f)) {
                ok = mbar_wait(o_full + (t - 1) % NBUF, ((t - 1) / NBUF) & 1, abort_flag, p.status, 421);
                if (!__all_sync(0xffffffffu, ok)) goto done;
                tc_fence_after();
#pragma unroll 1
                for (int c = 0; c < HD; c += 32) {
                  tmem_ld32(t_o + c, pk);
                  tmem_ld_wait(pk);
#pragma unroll
                  for (int e = 0; e < 32; ++e) pk[e] = __float_as_uint(__uint_as_float(pk[e]) * alpha);
                  tmem_st32(t_o + c, pk);
                  tmem_st_wait();
                }
              }
            }
            const float m_use = m_ref == -INFINITY ? 0.f : m_ref;
            const float2 sc2 = make_float2(sc, sc), m2 = make_float2(-m_use, -m_use);
            float2 sum0 = make_float2(0.f, 0.f), sum1 = sum0;
#pragma unroll
            for (int e = 0; e < 16; ++e) {
              float2 x = fma2(make_float2(__uint_as_float(a[2 * e]), __uint_as_float(a[2 * e + 1])), sc2, m2);
              x = make_float2(ex2(x.x), ex2(x.y));
              if (e & 1) sum1 = add2(sum1, x); else sum0 = add2(sum0, x);
              pk[e] = pack_bf16(x.x, x.y);
            }
#pragma unroll
            for (int e = 0; e < 16; ++e) {
              float2 x = fma2(make_float2(__uint_as_float(b[2 * e]), __uint_as_float(b[2 * e + 1])), sc2, m2);
              x = make_float2(ex2(x.x), ex2(x.y));
              if (e & 1) sum1 = add2(sum1, x); else sum0 = add2(sum0, x);
              pk[16 + e] = pack_bf16(x.x, x.y);
            }
            sum = (sum0.x + sum0.y) + (sum1.x + sum1.y);
            retake = row_ok && sum > kRescaleSum;        // some score has outgrown the reference
            if (!__any_sync(0xffffffffu, retake)) break;
          }
          l += sum;
          // P over the scores it came from, where the second product reads it as its A operand
          tmem_st32(t_s, pk);
          tmem_st_wait();
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(p_full + buf);
      }
      if (!warp_ok) continue;
      // the item's last product (products complete in issue order, so all of them)
      if (kt_hi > kt_lo) {
        bool ok = mbar_wait(o_full + (t - 1) % NBUF, ((t - 1) / NBUF) & 1, abort_flag, p.status, 423);
        if (!__all_sync(0xffffffffu, ok)) goto done;
        tc_fence_after();
      }

      // ---- item epilogue: one output row per thread
      const int head = kvh * p.group + row % p.group;
      uint4* out_row = reinterpret_cast<uint4*>(p.out + (size_t)(q_row0 + tok) * p.Hq * HD + head * HD);
      auto store32 = [&](const float (&o)[32], float inv, uint4* dst) {
#pragma unroll
        for (int c = 0; c < 4; ++c)
          dst[c] = make_uint4(pack_bf16(o[8 * c] * inv, o[8 * c + 1] * inv), pack_bf16(o[8 * c + 2] * inv, o[8 * c + 3] * inv),
                              pack_bf16(o[8 * c + 4] * inv, o[8 * c + 5] * inv), pack_bf16(o[8 * c + 6] * inv, o[8 * c + 7] * inv));
      };
      if (n_split == 1) {
        const float inv = 1.f / l;
#pragma unroll 1
        for (int c0 = 0; c0 < HD; c0 += 32) {              // (a whole warp reads tensor memory together)
          uint32_t u[32];
          tmem_ld32(t_o + c0, u);
          tmem_ld_wait(u);
          if (row_ok) {
            float o[32];
#pragma unroll
            for (int e = 0; e < 32; ++e) o[e] = __uint_as_float(u[e]);
            store32(o, inv, out_row + c0 / 8);
          }
        }
        tc_fence_before();
      } else {
        // Partials of this (q-tile, kv head, quarter): per slice the 32 rows' exponent references (log2 units), their sums
        // under them, then the unnormalised outputs, four dims of a row together: a warp's accesses are 512 contiguous
        // bytes.  A quarter is handed over by itself: the warp whose slice arrives last combines its 32 rows, so the
        // CTA's warps do not wait for one another here.
        constexpr int PART = (2 + HD) * 32;
        auto slice = [&](int k) -> float* { return p.split_ws + (size_t)((slice_slot(ib.z, k, ib.w) * p.Hkv + kvh) * p.plan.quarters + quarter) * PART; };
        float* part = slice(split) + lane;
        part[0] = m_ref;
        part[32] = l;
#pragma unroll 1
        for (int c0 = 0; c0 < HD; c0 += 32) {
          uint32_t u[32];
          tmem_ld32(t_o + c0, u);
          tmem_ld_wait(u);
          float4* dst = reinterpret_cast<float4*>(part - lane + 64) + (c0 / 4) * 32 + lane;
#pragma unroll
          for (int v = 0; v < 8; ++v)
            dst[v * 32] = make_float4(__uint_as_float(u[4 * v]), __uint_as_float(u[4 * v + 1]), __uint_as_float(u[4 * v + 2]),
                                      __uint_as_float(u[4 * v + 3]));
        }
        tc_fence_before();
        __threadfence();
        __syncwarp();
        int arrived = 0;
        if (lane == 0) {
          int* ctr = p.plan.counters + (ib.z * p.Hkv + kvh) * p.plan.quarters + quarter;
          arrived = atomicAdd(ctr, 1);
          if (arrived == n_split - 1) *ctr = 0;          // ready for the next layer
        }
        if (__shfl_sync(0xffffffffu, arrived, 0) == n_split - 1) {
          __threadfence();
          // Slices in order, whatever the order they arrived in, under a reference that grows with them; what three slices
          // left is in flight at once.
#pragma unroll 1
          for (int c0 = 0; c0 < HD; c0 += 32) {
            float o[32], L = 0.f, M = -INFINITY;
#pragma unroll
            for (int e = 0; e < 32; ++e) o[e] = 0.f;
#pragma unroll 1
            for (int k = 0; k < n_split; k += 3) {
              float m[3], ls[3];
              float4 x[3][8];
#pragma unroll
              for (int j = 0; j < 3; ++j) {
                if (k + j >= n_split) {
                  m[j] = -INFINITY;
                  ls[j] = 0.f;
#pragma unroll
                  for (int v = 0; v < 8; ++v) x[j][v] = make_float4(0.f, 0.f, 0.f, 0.f);
                } else {
                  const float* ps = slice(k + j);
                  const float4* src = reinterpret_cast<const float4*>(ps + 64) + (c0 / 4) * 32 + lane;
                  m[j] = __ldcg(ps + lane);
                  ls[j] = __ldcg(ps + 32 + lane);
#pragma unroll
                  for (int v = 0; v < 8; ++v) x[j][v] = __ldcg(src + v * 32);
                }
              }
              const float M_new = fmaxf(fmaxf(M, m[0]), fmaxf(m[1], m[2]));
              const float old = M == -INFINITY ? 0.f : ex2(M - M_new);
              M = M_new;
              L *= old;
#pragma unroll
              for (int e = 0; e < 32; ++e) o[e] *= old;
#pragma unroll
              for (int j = 0; j < 3; ++j) {
                const float wgt = m[j] == -INFINITY ? 0.f : ex2(m[j] - M);
                L += wgt * ls[j];
#pragma unroll
                for (int v = 0; v < 8; ++v) {
                  o[4 * v] += wgt * x[j][v].x;
                  o[4 * v + 1] += wgt * x[j][v].y;
                  o[4 * v + 2] += wgt * x[j][v].z;
                  o[4 * v + 3] += wgt * x[j][v].w;
                }
              }
            }
            if (row_ok) store32(o, 1.f / L, out_row + c0 / 8);
          }
        }
      }
     }
    }
  }

done:
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    if (*abort_flag) __nanosleep(20000);
    tmem_dealloc(tmem_base, C::TMEM_COLS);
  }
}

int launch_attn_sm100(cudaStream_t st, const CUtensorMap& tmQ, const CUtensorMap& tmK, const CUtensorMap& tmV,
                      const AttnPlan& plan, const KvView& kv, const ModelDims& md, int layer, bf16* out, int device,
                      int* status, float* split_ws, const uint4* anc, bool pdl) {
  static bool attr_set[2][kMaxDevices] = {};       // the attribute is per kernel and device
  if (device < 0 || device >= kMaxDevices || (md.D != 64 && md.D != 128)) return -1;
  const int which = md.D == 128;
  if (!attr_set[which][device]) {
    const cudaError_t e =
        which ? cudaFuncSetAttribute(attn_sm100_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, AttnCfg<128>::SMEM)
              : cudaFuncSetAttribute(attn_sm100_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, AttnCfg<64>::SMEM);
    if (e != cudaSuccess) return -1;
    attr_set[which][device] = true;
  }
  AttnParams p;
  p.plan = plan;
  p.block_table = kv.block_table;
  p.max_blocks = kv.max_blocks;
  p.n_blocks = kv.n_blocks;
  p.Hq = md.Hq;
  p.Hkv = md.Hkv;
  p.group = md.group;
  p.layer = layer;
  p.out = out;
  p.split_ws = split_ws;
  p.anc = anc;
  p.status = status;
  if (which)
    return launch_kernel(attn_sm100_kernel<128>, dim3(plan.grid), dim3(kAttnThreads), AttnCfg<128>::SMEM, st, pdl, tmQ, tmK,
                         tmV, p);
  return launch_kernel(attn_sm100_kernel<64>, dim3(plan.grid), dim3(kAttnThreads), AttnCfg<64>::SMEM, st, pdl, tmQ, tmK, tmV, p);
}

}  // namespace hsd
