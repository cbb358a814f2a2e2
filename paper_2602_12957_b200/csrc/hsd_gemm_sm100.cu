// tcgen05 / TMEM GEMM for sm_100a:  C = A W^T,  A [M,K] bf16 (activations), W [n_out,K] bf16 (weights),
// fp32 accumulation in tensor memory, operands staged in shared memory by TMA (128-byte swizzle).
//
// One persistent CTA per SM walks work units (128 x BN output tile, optionally one slice of K), M fastest so
// CTAs running side by side share a weight tile through L2.  Warp roles:
//   warp 0      A producer: activation tile, one TMA box per 64-column sub-tile of a stage, of 16, 32, 64 or 128 rows by the
//               rows of the call (gemm_a_box_rows)
//   warp 1      MMA issuer and TMEM owner
//   warp 2      B producer: the two halves of the weight tile, one TMA box each per sub-tile (a pair's CTA: its half).
//               Weights do not depend on the previous kernel, so it starts before the programmatic-launch wait.
//   warps 4..7  epilogue, one TMEM lane quarter each (warp w works on lane quarter w mod 4, the hardware's rule)
// Warps 0 to 2 elect one lane that runs their whole loop.  With `elect` the compiler knows that one thread is active, and
// TMA and MMA instructions take their operands as they are; a lane chosen by its number paid ~0.25 us for a TMA
// instruction and ~90 cycles for an MMA, and an election at every stage ~70 cycles for each of a stage's narrow MMAs.
// Verification steps, election at every stage / once: 16 plain rows 0.910 / 0.893 ms, 136 rows 1.040 / 1.019 ms, 320 rows
// 1.658 / 1.636 ms, one lane's 128-node tree 1.200 / 1.182 ms.
// Two accumulator buffers in TMEM let the epilogue of unit i overlap the main loop of unit i+1.
//
// Epilogues (all fused; results leave the SM through swizzled staging buffers and TMA stores, so global
// writes are full 128-byte lines whatever the thread-to-row mapping in TMEM):
//   GS_STORE_BF16  C bf16 = acc
//   GS_ADD_F32     C fp32 += acc   (TMA reduce-add into the residual stream; with split-K every K slice adds)
//   GS_SWIGLU      C bf16 = silu(gate) * up              (gate rows and up rows of W land in one tile)
//   GS_ARGMAX      per-row running argmax over the vocabulary + the next draft token's logit; logits never
//                  leave the SM (Eq. 10 of the paper fused into the LM head)
//   GS_QKV_ROPE    rotary embedding on q and k heads, q -> packed bf16, k/v -> paged KV pool (head_dim 64;
//                  GS_QKV_ROPE128: the same for head_dim 128)
#include <atomic>

#include "hsd_kernels.h"

namespace hsd {

// ------------------------------------------------------------------------------------------------
// driver entry point for tensor-map encoding (resolved at run time; the library does not link libcuda)
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
static EncodeTiledFn g_encode = nullptr;

int tma_init() {
  if (g_encode) return 0;
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult qres;
  cudaError_t e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres);
  if (e != cudaSuccess || qres != cudaDriverEntryPointSuccess || !fn) return -1;
  g_encode = reinterpret_cast<EncodeTiledFn>(fn);
  return 0;
}

int make_tmap_2d(CUtensorMap* map, const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows) {
  if (!g_encode) return -1;
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {cols * 2};
  cuuint32_t box[2] = {64, box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? 0 : -1;
}

int make_tmap_2d_f32(CUtensorMap* map, const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows) {
  if (!g_encode) return -1;
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {cols * 4};
  cuuint32_t box[2] = {32, box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = g_encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(base), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? 0 : -1;
}

int make_tmap_3d(CUtensorMap* map, const void* base, uint64_t d0, uint64_t d1, uint64_t d2, uint64_t stride1_bytes,
                 uint64_t stride2_bytes, uint32_t b0, uint32_t b1, uint32_t b2) {
  if (!g_encode) return -1;
  cuuint64_t dims[3] = {d0, d1, d2};
  cuuint64_t strides[2] = {stride1_bytes, stride2_bytes};
  cuuint32_t box[3] = {b0, b1, b2};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? 0 : -1;
}

// ------------------------------------------------------------------------------------------------
constexpr int BM = 128;
constexpr int KSUB = 64;                         // one 128-byte-swizzled sub-tile spans 64 bf16 of K
constexpr int kGemmThreads = 256;
constexpr int STG_BYTES = 4096;                  // one epilogue staging buffer: 32 rows x 128 bytes
constexpr int STG_TOTAL = 4 * 2 * STG_BYTES;     // four epilogue warps, two buffers each

// PAIR: two CTAs (a cluster) share one 256 x BN tile: each stages its own 128 rows of A and BN/2 rows of B.
// KSTEPS: sub-tiles of a stage.  A stage is one barrier round trip of ~250 cycles.  The MMAs or the fill of the 128- and
// 256-wide tiles' stages cover it (two sub-tiles: 256 wide the same, 128 wide 1 % slower steps, fewer stages being in
// flight), those of the 64-wide tile do not: plain decode 0.965 -> 0.947 ms, short drafts 1.059 -> 1.046 with two.
// ROWS: rows of A a stage has room for.  A call of at most 16 or 64 rows has its own kernels for the 64-wide tile: the MMA
// takes 128 rows all the same, and reads beyond a sub-tile's ROWS whatever lies behind it in the stage (rows are independent,
// and those go nowhere), but 18 or 12 k-blocks are under way in place of 8.  Steps of 16 plain rows 868 -> 861 us (gate/up 6.8 ->
// 6.5 us a launch, QKV 5.8 -> 5.55); what is left of the loop is the MMAs, whose 128 rows of A cost 32 cycles of shared memory each.
template <int BN, bool PAIR, int ROWS>
struct Cfg {
  static constexpr int A_SUB = ROWS * KSUB * 2;                     // bytes of one A sub-tile
  static constexpr int KSTEPS = BN == 64 ? 2 : 1;
  static constexpr int BK = KSUB * KSTEPS;                          // K extent of one stage
  static constexpr int A_BYTES = A_SUB * KSTEPS;
  static constexpr int B_SUB = (PAIR ? BN / 2 : BN) * KSUB * 2;     // bytes of one B sub-tile this CTA stages
  static constexpr int B_BYTES = B_SUB * KSTEPS;                    // bytes of B per stage
  static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr int STAGES = 192 * 1024 / STAGE_BYTES < 9 ? 192 * 1024 / STAGE_BYTES : BN == 64 ? 9 : 8;
  static constexpr int TMEM_COLS = BN <= 64 ? 128 : BN <= 128 ? 256 : 512;      // two accumulators, a power of two
  static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + STG_TOTAL + 1024 /*alignment slack*/ + 256 /*barriers*/;
};

struct GemmDev {
  int M, n_cols, K, n_up_off;   // n_cols: output columns; n_up_off: row offset of the `up` half (SwiGLU)
  int splits, kb_per_split;     // K slices per tile (GS_ADD_F32 only) and k-blocks per slice
  int a_box;                    // rows of an activation box (< 128 only where M is no more than that)
  GemmOut out;
  QkvEpilogue qkv;
  int* status;
};

// TMA store / reduce of one staging buffer and the bulk-group bookkeeping around it (issued by one lane).
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, const void* smem_src, int x, int y) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];"
               ::"l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(smem_src)), "r"(x), "r"(y)
               : "memory");
}
__device__ __forceinline__ void tma_reduce_add_2d(const CUtensorMap* map, const void* smem_src, int x, int y) {
  asm volatile("cp.reduce.async.bulk.tensor.2d.global.shared::cta.add.bulk_group [%0, {%2, %3}], [%1];"
               ::"l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(smem_src)), "r"(x), "r"(y)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void bulk_wait_read() {
  asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}


// 16-byte chunk `c` of this lane's 128-byte staging row, at its 128-byte-swizzle position.
__device__ __forceinline__ uint4* stg_chunk(uint8_t* buf, int lane, int c) {
  return reinterpret_cast<uint4*>(buf + lane * 128 + ((c ^ (lane & 7)) << 4));
}
__device__ __forceinline__ uint4 pack8(const uint32_t* r) {
  uint4 o;
  o.x = pack_bf16(__uint_as_float(r[0]), __uint_as_float(r[1]));
  o.y = pack_bf16(__uint_as_float(r[2]), __uint_as_float(r[3]));
  o.z = pack_bf16(__uint_as_float(r[4]), __uint_as_float(r[5]));
  o.w = pack_bf16(__uint_as_float(r[6]), __uint_as_float(r[7]));
  return o;
}

template <int BN, int MODE, bool PAIR, int ROWS>
__global__ void __launch_bounds__(kGemmThreads, 1)
gemm_sm100_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                  const __grid_constant__ CUtensorMap tmC, GemmDev p) {
  using C = Cfg<BN, PAIR, ROWS>;
  static_assert((C::KSTEPS - 1) * C::A_SUB + BM * KSUB * 2 <= C::STAGE_BYTES, "an MMA reads 128 rows from every sub-tile on");
  constexpr int KSTEPS = C::KSTEPS, BK = C::BK, A_BYTES = C::A_BYTES, A_SUB = C::A_SUB;
  constexpr int OUT_N = (MODE == GS_SWIGLU) ? BN / 2 : BN;   // output columns per tile
  constexpr int HALF_B = BN / 2 * KSUB * 2;                  // bytes of one weight half-tile of one sub-tile
  constexpr int TILE_M = PAIR ? 2 * BM : BM;                 // rows of one work unit (both CTAs of a pair)
  const int rank = PAIR ? (int)cluster_ctarank() : 0;        // 0 = the CTA that issues the MMAs
  const int cta = PAIR ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;       // index among the unit walkers
  const int n_cta = PAIR ? (int)(gridDim.x >> 1) : (int)gridDim.x;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* stg = smem + C::STAGES * C::STAGE_BYTES;
  uint64_t* bars = reinterpret_cast<uint64_t*>(stg + STG_TOTAL);
  uint64_t* full = bars;
  uint64_t* empty = bars + C::STAGES;
  uint64_t* tfull = bars + 2 * C::STAGES;
  uint64_t* tempty = tfull + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tempty + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < C::STAGES; ++s) {
      // A producer and B producer, each with its own byte count; a pair: one arrival (even CTA) for all bytes
      mbar_init(full + s, PAIR ? 1 : 2);
      mbar_init(empty + s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(tfull + b, 1);
      mbar_init(tempty + b, PAIR ? 8 : 4);     // the epilogue warps of both CTAs release the even CTA's MMA thread
    }
    *abort_flag = 0;
    fence_mbar_init();
    tma_prefetch_desc(&tmA);
    tma_prefetch_desc(&tmB);
    if (MODE != GS_ARGMAX) tma_prefetch_desc(&tmC);
  }
  if (warp == 1) {
    if (PAIR) {
      tmem_alloc_pair(tmem_slot, C::TMEM_COLS);
      tmem_relinquish_pair();
    } else {
      tmem_alloc(tmem_slot, C::TMEM_COLS);
      tmem_relinquish();
    }
  }
  tc_fence_before();
  __syncthreads();
  if (PAIR) cluster_sync();          // both CTAs' barriers exist before either one's loads complete on them
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  const int m_tiles = (p.M + TILE_M - 1) / TILE_M;
  const int n_tiles = (p.n_cols + OUT_N - 1) / OUT_N;      // (96, 160, 192 and 224 columns: the last tile may reach beyond)
  const int tiles = m_tiles * n_tiles;
  const int total = tiles * p.splits;
  const int k_blocks = (p.K + BK - 1) / BK;      // (a last stage beyond K is filled with zeros)

  // kc counts k-blocks over all units of this CTA: stage = kc % C::STAGES, the barriers' parities follow
  if (warp == 0) {
    // ---- A producer: activations, written by the previous kernel
    if (elect_one()) {
      pdl_wait();
      pdl_launch_dependents();
      int s = 0;
      uint32_t ph = 1;
      for (int t = cta; t < total; t += n_cta) {
        const int tile = t % tiles, split = t / tiles;
        const int m0 = (tile % m_tiles) * TILE_M + rank * BM;
        const int kb0 = split * p.kb_per_split, kb1 = min(k_blocks, kb0 + p.kb_per_split);
        for (int kb = kb0; kb < kb1; ++kb) {
          if (!mbar_wait(empty + s, ph, abort_flag, p.status, 100)) goto done;
          uint8_t* dst = smem + s * C::STAGE_BYTES;
          if (PAIR) {
            if (rank == 0) mbar_expect_tx(full + s, 2 * C::STAGE_BYTES);   // A and B of both CTAs land on this barrier
#pragma unroll
            for (int u = 0; u < KSTEPS; ++u) tma_load_2d_pair(dst + u * A_SUB, &tmA, full + s, kb * BK + u * KSUB, m0);
          } else {
            mbar_expect_tx(full + s, p.a_box * (KSUB * 2) * KSTEPS);
#pragma unroll
            for (int u = 0; u < KSTEPS; ++u) tma_load_2d(dst + u * A_SUB, &tmA, full + s, kb * BK + u * KSUB, m0);
          }
          if (++s == C::STAGES) { s = 0; ph ^= 1u; }
        }
      }
    }
  } else if (warp == 2) {
    // ---- B producer: both halves of the weight tile (for SwiGLU: gate rows / up rows); a pair's CTA stages half `rank`
    if (elect_one()) {
      int s = 0;
      uint32_t ph = 1;
      for (int t = cta; t < total; t += n_cta) {
        const int tile = t % tiles, split = t / tiles;
        const int n0 = (tile / m_tiles) * OUT_N;
        const int kb0 = split * p.kb_per_split, kb1 = min(k_blocks, kb0 + p.kb_per_split);
        const int row0 = n0, row1 = (MODE == GS_SWIGLU) ? p.n_up_off + n0 : n0 + BN / 2;
        for (int kb = kb0; kb < kb1; ++kb) {
          if (!mbar_wait(empty + s, ph, abort_flag, p.status, 110)) goto done;
          uint8_t* dst = smem + s * C::STAGE_BYTES + A_BYTES;
          if (PAIR) {
#pragma unroll
            for (int u = 0; u < KSTEPS; ++u)
              tma_load_2d_pair(dst + u * C::B_SUB, &tmB, full + s, kb * BK + u * KSUB, rank ? row1 : row0);
          } else {
            mbar_expect_tx(full + s, C::B_BYTES);
#pragma unroll
            for (int u = 0; u < KSTEPS; ++u) {
              tma_load_2d(dst + u * C::B_SUB, &tmB, full + s, kb * BK + u * KSUB, row0);
              tma_load_2d(dst + u * C::B_SUB + HALF_B, &tmB, full + s, kb * BK + u * KSUB, row1);
            }
          }
          if (++s == C::STAGES) { s = 0; ph ^= 1u; }
        }
      }
    }
  } else if (warp == 1) {
    if (rank == 0 && elect_one()) {
      constexpr uint32_t idesc = umma_idesc_bf16(BN, false, TILE_M);
      const uint64_t desc0 = umma_desc_sw128(smem_u32(smem));      // a byte offset adds a sixteenth of itself
      int s = 0;
      uint32_t ph = 0;
      int it = 0;
      for (int t = cta; t < total; t += n_cta, ++it) {
        const int split = t / tiles;
        const int kb0 = split * p.kb_per_split, kb1 = min(k_blocks, kb0 + p.kb_per_split);
        const int b = it & 1;
        const uint32_t aph = (it >> 1) & 1;
        if (!mbar_wait(tempty + b, aph ^ 1u, abort_flag, p.status, 200)) goto done;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + b * BN;
        for (int kb = kb0; kb < kb1; ++kb) {
          if (!mbar_wait(full + s, ph, abort_flag, p.status, 201)) goto done;
          tc_fence_after();
          const uint64_t da = desc0 + s * (C::STAGE_BYTES / 16), db = da + A_BYTES / 16;
#pragma unroll
          for (int u = 0; u < KSTEPS; ++u) {
#pragma unroll
            for (int k = 0; k < KSUB / 16; ++k) {
              const uint32_t acc = (kb != kb0 || u != 0 || k != 0) ? 1u : 0u;
              if (PAIR) umma_bf16_pair(d_tmem, da + (u * A_SUB + k * 32) / 16, db + (u * C::B_SUB + k * 32) / 16, idesc, acc);
              else umma_bf16(d_tmem, da + (u * A_SUB + k * 32) / 16, db + (u * C::B_SUB + k * 32) / 16, idesc, acc);
            }
          }
          // smem stage reusable once these MMAs have read it (in both CTAs of a pair)
          if (PAIR) umma_commit_pair(empty + s); else umma_commit(empty + s);
          if (kb + 1 == kb1) {                                   // accumulator complete
            if (PAIR) umma_commit_pair(tfull + b); else umma_commit(tfull + b);
          }
          if (++s == C::STAGES) { s = 0; ph ^= 1u; }
        }
      }
    }
  } else if (warp >= 4) {
    // ---- epilogue warps 4..7
    const int quarter = warp & 3;                 // TMEM lanes [32*quarter, +32) belong to this warp
    const int row_in_tile = quarter * 32 + lane;
    uint8_t* my_stg = stg + quarter * 2 * STG_BYTES;
    int n_stores = 0;                             // staging buffers handed to TMA so far (selects the buffer)
    pdl_wait();
    int it = 0;
    for (int t = cta; t < total; t += n_cta, ++it) {
      const int b = it & 1;
      const uint32_t aph = (it >> 1) & 1;
      const int tile = t % tiles;
      const int m0 = (tile % m_tiles) * TILE_M + rank * BM, n0 = (tile / m_tiles) * OUT_N;
      const int row = m0 + row_in_tile;
      const bool row_ok = row < p.M;
      const int wrow0 = m0 + quarter * 32;        // first row of this warp's 32-row slab
      const bool slab_ok = wrow0 < p.M;           // warp-uniform: the slab has at least one real row
      // rotary (cos, sin) of this thread's row: fetched while the main loop still runs, reused by every head
      float4 cs[MODE == GS_QKV_ROPE ? 16 : 1];
      if (MODE == GS_QKV_ROPE && row_ok) {
        const float4* src = reinterpret_cast<const float4*>(p.qkv.rope_cs + (size_t)row * 32);
#pragma unroll
        for (int i = 0; i < 16; ++i) cs[i] = __ldg(src + i);
      }
      // likewise the two words the K/V stores depend on (read here, used after the accumulator is ready).  row_kv
      // comes from the step's set-up kernel: after a failed device-side check it was not written, so nothing is
      // stored through it (q included: the step is a no-op), nor through a row outside the pool
      bool live = true;
      int phys = 0;
      int nxt = -1;                                 // LM head: the row's next draft token (its logit is captured)
      if (MODE == GS_ARGMAX) nxt = (row_ok && p.out.row_next) ? p.out.row_next[row] : -1;
      if (MODE == GS_QKV_ROPE || MODE == GS_QKV_ROPE128) {
        const int st_word = p.status ? *p.status : 0;
        const int kv_row = row_ok ? p.qkv.row_kv[row] : 0;
        live = st_word == 0;
        phys = live ? kv_row : 0;
      }
      bool ok = mbar_wait(tfull + b, aph, abort_flag, p.status, 300);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) goto done;
      tc_fence_after();
      const uint32_t t_acc = tmem_base + (uint32_t(quarter * 32) << 16) + b * BN;

      // A slab wholly beyond M stages nothing: every staged chunk commits exactly one bulk group, which is what
      // lets "at most one group pending" protect the buffer about to be rewritten.
      if (MODE == GS_STORE_BF16) {
#pragma unroll 1
        for (int c = 0; slab_ok && c < BN && n0 + c < p.n_cols; c += 64) {
          uint8_t* buf = my_stg + (n_stores & 1) * STG_BYTES;
          if (lane == 0) bulk_wait_read<1>();      // the store that last read this buffer has drained
          __syncwarp();
          uint32_t r0[32], r1[32];
          tmem_ld32(t_acc + c, r0);
          tmem_ld32(t_acc + c + 32, r1);
          tmem_ld_wait();
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            *stg_chunk(buf, lane, v) = pack8(r0 + 8 * v);
            *stg_chunk(buf, lane, 4 + v) = pack8(r1 + 8 * v);
          }
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) {
            tma_store_2d(&tmC, buf, n0 + c, wrow0);
            bulk_commit();
          }
          ++n_stores;
        }
      } else if (MODE == GS_ADD_F32) {
#pragma unroll 1
        for (int c = 0; slab_ok && c < BN && n0 + c < p.n_cols; c += 32) {
          uint8_t* buf = my_stg + (n_stores & 1) * STG_BYTES;
          if (lane == 0) bulk_wait_read<1>();
          __syncwarp();
          uint32_t r[32];
          tmem_ld32(t_acc + c, r);
          tmem_ld_wait();
#pragma unroll
          for (int v = 0; v < 8; ++v)
            *stg_chunk(buf, lane, v) = make_uint4(r[4 * v], r[4 * v + 1], r[4 * v + 2], r[4 * v + 3]);
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) {
            tma_reduce_add_2d(&tmC, buf, n0 + c, wrow0);
            bulk_commit();
          }
          ++n_stores;
        }
      } else if (MODE == GS_SWIGLU && OUT_N == 32) {
        // the narrow tile: a row's 32 outputs are 64 bytes, stored as they are
        if (slab_ok) {
          uint32_t g[32], u[32];
          tmem_ld32(t_acc, g);
          tmem_ld32(t_acc + OUT_N, u);
          tmem_ld_wait();
#pragma unroll
          for (int e = 0; e < 32; ++e) {
            const float gv = __uint_as_float(g[e]);
            g[e] = __float_as_uint(__fdividef(gv, 1.f + __expf(-gv)) * __uint_as_float(u[e]));
          }
          if (row_ok) {
            uint4* dst = reinterpret_cast<uint4*>(static_cast<bf16*>(p.out.C) + (size_t)row * p.out.ldc + n0);
#pragma unroll
            for (int v = 0; v < 4; ++v) dst[v] = pack8(g + 8 * v);
          }
        }
      } else if (MODE == GS_SWIGLU) {
#pragma unroll 1
        for (int c = 0; slab_ok && c + 64 <= OUT_N; c += 64) {
          uint8_t* buf = my_stg + (n_stores & 1) * STG_BYTES;
          if (lane == 0) bulk_wait_read<1>();
          __syncwarp();
#pragma unroll
          for (int hf = 0; hf < 2; ++hf) {
            uint32_t g[32], u[32];
            tmem_ld32(t_acc + c + hf * 32, g);
            tmem_ld32(t_acc + OUT_N + c + hf * 32, u);
            tmem_ld_wait();
#pragma unroll
            for (int e = 0; e < 32; ++e) {
              // silu(g) * u; the approximate divide (reciprocal + multiply, 2 ulp) has no slow-path branch, so the
              // 32 elements interleave; the result is rounded to bf16 anyway
              const float gv = __uint_as_float(g[e]);
              g[e] = __float_as_uint(__fdividef(gv, 1.f + __expf(-gv)) * __uint_as_float(u[e]));
            }
#pragma unroll
            for (int v = 0; v < 4; ++v) *stg_chunk(buf, lane, hf * 4 + v) = pack8(g + 8 * v);
          }
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) {
            tma_store_2d(&tmC, buf, n0 + c, wrow0);
            bulk_commit();
          }
          ++n_stores;
        }
        // what is left of 80, 96 or 112 outputs: whole 32-byte sectors, stored as they are
#pragma unroll 1
        for (int c = OUT_N / 64 * 64; OUT_N % 64 && slab_ok && c < OUT_N && n0 + c < p.n_cols; c += 16) {
          uint32_t g[16], u[16];
          tmem_ld16(t_acc + c, g);
          tmem_ld16(t_acc + OUT_N + c, u);
          tmem_ld_wait(g);
          tmem_ld_wait(u);
#pragma unroll
          for (int e = 0; e < 16; ++e) {
            const float gv = __uint_as_float(g[e]);
            g[e] = __float_as_uint(__fdividef(gv, 1.f + __expf(-gv)) * __uint_as_float(u[e]));
          }
          if (row_ok) {
            uint4* dst = reinterpret_cast<uint4*>(static_cast<bf16*>(p.out.C) + (size_t)row * p.out.ldc + n0 + c);
            dst[0] = pack8(g);
            dst[1] = pack8(g + 8);
          }
        }
      } else if (MODE == GS_ARGMAX) {
        float best_v = -INFINITY, zd = 0.f;
        int best_c = n0;
#pragma unroll 1
        for (int c = 0; c < BN; c += 32) {
          uint32_t r[32];
          tmem_ld32(t_acc + c, r);
          tmem_ld_wait();
#pragma unroll
          for (int e = 0; e < 32; ++e) {
            const float v = __uint_as_float(r[e]);
            const int col = n0 + c + e;
            if (v > best_v) { best_v = v; best_c = col; }
            if (col == nxt) zd = v;
          }
        }
        if (row_ok) {
          atomicMax(p.out.row_best + row, argmax_key(best_v, best_c));
          if (nxt >= n0 && nxt < n0 + BN) p.out.zdraft[row] = zd;
        }
      } else if (MODE == GS_QKV_ROPE) {
        const bool kv_ok = live && phys >= 0 && phys < p.qkv.kv_rows;
        if (!kv_ok) phys = 0;
        const int blk = phys >> 6, off = phys & 63;
#pragma unroll 1
        for (int hh = 0; hh < BN / 64; ++hh) {
          const int head = n0 / 64 + hh;
          const bool is_q = head < p.qkv.Hq;
          if (!slab_ok || head >= p.qkv.Hq + 2 * p.qkv.Hkv) break;
          uint8_t* buf = my_stg + (n_stores & 1) * STG_BYTES;
          if (is_q) {
            if (lane == 0) bulk_wait_read<1>();
            __syncwarp();
          }
          uint32_t lo[32], hi[32];
          tmem_ld32(t_acc + hh * 64, lo);
          tmem_ld32(t_acc + hh * 64 + 32, hi);
          tmem_ld_wait();
          if (p.qkv.q_norm && head < p.qkv.Hq + p.qkv.Hkv && row_ok) {
            // per-head RMSNorm of q and k over the head's 64 dims (all in this thread) before the rotation
            float ss = 0.f;
#pragma unroll
            for (int i = 0; i < 32; ++i)
              ss += __uint_as_float(lo[i]) * __uint_as_float(lo[i]) + __uint_as_float(hi[i]) * __uint_as_float(hi[i]);
            const float rs = rsqrtf(ss * (1.f / 64.f) + p.qkv.eps);
            const uint4* g4 = reinterpret_cast<const uint4*>(is_q ? p.qkv.q_norm : p.qkv.k_norm);
#pragma unroll
            for (int v = 0; v < 4; ++v) {
              const uint4 gl = __ldg(g4 + v), gh = __ldg(g4 + 4 + v);
              const uint32_t wl[4] = {gl.x, gl.y, gl.z, gl.w}, wh[4] = {gh.x, gh.y, gh.z, gh.w};
#pragma unroll
              for (int k = 0; k < 4; ++k) {
                lo[8 * v + 2 * k] = __float_as_uint(__uint_as_float(lo[8 * v + 2 * k]) * rs * bf16_lo(wl[k]));
                lo[8 * v + 2 * k + 1] = __float_as_uint(__uint_as_float(lo[8 * v + 2 * k + 1]) * rs * bf16_hi(wl[k]));
                hi[8 * v + 2 * k] = __float_as_uint(__uint_as_float(hi[8 * v + 2 * k]) * rs * bf16_lo(wh[k]));
                hi[8 * v + 2 * k + 1] = __float_as_uint(__uint_as_float(hi[8 * v + 2 * k + 1]) * rs * bf16_hi(wh[k]));
              }
            }
          }
          if (head < p.qkv.Hq + p.qkv.Hkv && row_ok) {
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              const float4 c2 = cs[i];   // (cos, sin) of frequencies 2i and 2i+1
              const float a0 = __uint_as_float(lo[2 * i]), b0 = __uint_as_float(hi[2 * i]);
              const float a1 = __uint_as_float(lo[2 * i + 1]), b1 = __uint_as_float(hi[2 * i + 1]);
              lo[2 * i] = __float_as_uint(a0 * c2.x - b0 * c2.y);
              hi[2 * i] = __float_as_uint(b0 * c2.x + a0 * c2.y);
              lo[2 * i + 1] = __float_as_uint(a1 * c2.z - b1 * c2.w);
              hi[2 * i + 1] = __float_as_uint(b1 * c2.z + a1 * c2.w);
            }
          }
          if (is_q) {
#pragma unroll
            for (int v = 0; v < 4; ++v) {
              *stg_chunk(buf, lane, v) = pack8(lo + 8 * v);
              *stg_chunk(buf, lane, 4 + v) = pack8(hi + 8 * v);
            }
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0 && live) {
              tma_store_2d(&tmC, buf, head * 64, wrow0);
              bulk_commit();
            }
            ++n_stores;
          } else if (row_ok && kv_ok) {
            // K and V rows go to the paged pool: one 128-byte line per (token, kv head)
            const bool is_k = head < p.qkv.Hq + p.qkv.Hkv;
            bf16* pool = is_k ? p.qkv.k_pool_layer : p.qkv.v_pool_layer;
            const int kvh = head - p.qkv.Hq - (is_k ? 0 : p.qkv.Hkv);
            uint4* d4 = reinterpret_cast<uint4*>(pool + (((size_t)blk * p.qkv.Hkv + kvh) * 64 + off) * 64);
#pragma unroll
            for (int v = 0; v < 4; ++v) {
              d4[v] = pack8(lo + 8 * v);
              d4[4 + v] = pack8(hi + 8 * v);
            }
          }
        }
      }
      else if (MODE == GS_QKV_ROPE128) {
        // head_dim 128: a head is 128 accumulator columns and the rotation pairs dim i with dim i + 64, so a head is
        // worked in two passes of 32 pairs (columns [32c, 32c+32) with [64+32c, 64+32c+32)); the row's (cos, sin) of
        // those 32 frequencies come from the table per pass.  q leaves through two staging buffers (dims 0..63 and
        // 64..127), both filled by the two passes and stored together.
        const bool kv_ok = live && phys >= 0 && phys < p.qkv.kv_rows;
        if (!kv_ok) phys = 0;
        const int blk = phys >> 6, off = phys & 63;
#pragma unroll 1
        for (int hh = 0; hh < BN / 128; ++hh) {
          const int head = n0 / 128 + hh;
          const bool is_q = head < p.qkv.Hq;
          const bool rot = head < p.qkv.Hq + p.qkv.Hkv;           // q and k heads are normalised (if asked) and rotated
          if (!slab_ok) break;
          float rs = 1.f;
          // (warp-uniform: a tensor-memory load is executed by the whole warp, rows beyond M included)
          const bool normed = p.qkv.q_norm && rot;
          if (normed) {                                            // per-head RMSNorm over the head's 128 dims
            float ss = 0.f;
#pragma unroll 1
            for (int c = 0; c < 4; ++c) {
              uint32_t r[32];
              tmem_ld32(t_acc + hh * 128 + c * 32, r);
              tmem_ld_wait();
#pragma unroll
              for (int i = 0; i < 32; ++i) ss += __uint_as_float(r[i]) * __uint_as_float(r[i]);
            }
            rs = rsqrtf(ss * (1.f / 128.f) + p.qkv.eps);
          }
          if (is_q) {
            if (lane == 0) bulk_wait_read<0>();                    // both staging buffers are free
            __syncwarp();
          }
          const bool is_k = rot && !is_q;
          bf16* pool = is_k ? p.qkv.k_pool_layer : p.qkv.v_pool_layer;
          const int kvh = head - p.qkv.Hq - (is_k || is_q ? 0 : p.qkv.Hkv);
          uint4* d4 = reinterpret_cast<uint4*>(pool + (((size_t)blk * p.qkv.Hkv + (is_q ? 0 : kvh)) * 64 + off) * 128);
#pragma unroll 1
          for (int c = 0; c < 2; ++c) {
            uint32_t lo[32], hi[32];
            tmem_ld32(t_acc + hh * 128 + c * 32, lo);
            tmem_ld32(t_acc + hh * 128 + 64 + c * 32, hi);
            tmem_ld_wait();
            if (normed && row_ok) {
              const uint4* g4 = reinterpret_cast<const uint4*>(is_q ? p.qkv.q_norm : p.qkv.k_norm);
#pragma unroll
              for (int v = 0; v < 4; ++v) {
                const uint4 gl = __ldg(g4 + 4 * c + v), gh = __ldg(g4 + 8 + 4 * c + v);
                const uint32_t wl[4] = {gl.x, gl.y, gl.z, gl.w}, wh[4] = {gh.x, gh.y, gh.z, gh.w};
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                  lo[8 * v + 2 * k] = __float_as_uint(__uint_as_float(lo[8 * v + 2 * k]) * rs * bf16_lo(wl[k]));
                  lo[8 * v + 2 * k + 1] = __float_as_uint(__uint_as_float(lo[8 * v + 2 * k + 1]) * rs * bf16_hi(wl[k]));
                  hi[8 * v + 2 * k] = __float_as_uint(__uint_as_float(hi[8 * v + 2 * k]) * rs * bf16_lo(wh[k]));
                  hi[8 * v + 2 * k + 1] = __float_as_uint(__uint_as_float(hi[8 * v + 2 * k + 1]) * rs * bf16_hi(wh[k]));
                }
              }
            }
            if (rot && row_ok) {
              const float4* src = reinterpret_cast<const float4*>(p.qkv.rope_cs + (size_t)row * 64 + c * 32);
#pragma unroll
              for (int i = 0; i < 16; ++i) {
                const float4 c2 = __ldg(src + i);   // (cos, sin) of frequencies 32c + 2i and 32c + 2i + 1
                const float a0 = __uint_as_float(lo[2 * i]), b0 = __uint_as_float(hi[2 * i]);
                const float a1 = __uint_as_float(lo[2 * i + 1]), b1 = __uint_as_float(hi[2 * i + 1]);
                lo[2 * i] = __float_as_uint(a0 * c2.x - b0 * c2.y);
                hi[2 * i] = __float_as_uint(b0 * c2.x + a0 * c2.y);
                lo[2 * i + 1] = __float_as_uint(a1 * c2.z - b1 * c2.w);
                hi[2 * i + 1] = __float_as_uint(b1 * c2.z + a1 * c2.w);
              }
            }
            if (is_q) {
#pragma unroll
              for (int v = 0; v < 4; ++v) {
                *stg_chunk(my_stg, lane, 4 * c + v) = pack8(lo + 8 * v);
                *stg_chunk(my_stg + STG_BYTES, lane, 4 * c + v) = pack8(hi + 8 * v);
              }
            } else if (row_ok && kv_ok) {
              // K and V rows go to the paged pool: one 256-byte row per (token, kv head)
#pragma unroll
              for (int v = 0; v < 4; ++v) {
                d4[4 * c + v] = pack8(lo + 8 * v);
                d4[8 + 4 * c + v] = pack8(hi + 8 * v);
              }
            }
          }
          if (is_q) {
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0 && live) {
              tma_store_2d(&tmC, my_stg, head * 128, wrow0);
              tma_store_2d(&tmC, my_stg + STG_BYTES, head * 128 + 64, wrow0);
              bulk_commit();
            }
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (PAIR) mbar_arrive_even_cta(tempty + b); else mbar_arrive(tempty + b);
      }
    }
    if (lane == 0) bulk_wait_all();               // staged rows have reached global memory (waiting only for the
                                                  // staging reads measured no shorter)
  }

done:
  tc_fence_before();
  __syncthreads();
  if (PAIR) cluster_sync();                // the other CTA's loads, MMAs and arrivals no longer touch this one
  if (warp == 1) {
    if (*abort_flag) __nanosleep(20000);   // let copies / MMAs in flight drain before TMEM goes away
    if (PAIR) tmem_dealloc_pair(tmem_base, C::TMEM_COLS); else tmem_dealloc(tmem_base, C::TMEM_COLS);
  }
}

// ------------------------------------------------------------------------------------------------
template <int BN, int MODE, bool PAIR, int ROWS = BM>
static int launch_one(cudaStream_t st, const GemmSm100Args& a, int splits) {
  using C = Cfg<BN, PAIR, ROWS>;
  constexpr int OUT_N = (MODE == GS_SWIGLU) ? BN / 2 : BN;
  GemmDev p;
  p.M = a.M;
  p.K = a.K;
  p.n_cols = (MODE == GS_SWIGLU) ? a.n_out / 2 : a.n_out;
  p.n_up_off = a.n_out / 2;
  const int k_blocks = (a.K + C::BK - 1) / C::BK;
  while (splits > 1 && (splits - 1) * ((k_blocks + splits - 1) / splits) >= k_blocks) --splits;    // no slice is empty
  p.splits = splits;
  p.kb_per_split = (k_blocks + splits - 1) / splits;
  p.a_box = (int)gemm_a_box_rows(a.M);
  p.out = a.out;
  p.qkv = a.qkv;
  p.status = a.status;
  const int tile_m = PAIR ? 2 * BM : BM;
  const int m_tiles = (a.M + tile_m - 1) / tile_m;
  const int total = m_tiles * ((p.n_cols + OUT_N - 1) / OUT_N) * splits;
  const int walkers = PAIR ? a.n_sms / 2 : a.n_sms;
  const int grid = (total < walkers ? total : walkers) * (PAIR ? 2 : 1);
  const CUtensorMap& tmB = a.tmB->half_tile(BN);      // (a pair's CTA loads one box, others two)
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kGemmThreads);
  cfg.dynamicSmemBytes = C::SMEM_BYTES;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  int n_attr = 0;
  if (a.pdl) {
    attr[n_attr].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n_attr].val.programmaticStreamSerializationAllowed = 1;
    ++n_attr;
  }
  if (PAIR) {
    attr[n_attr].id = cudaLaunchAttributeClusterDimension;
    attr[n_attr].val.clusterDim.x = 2;
    attr[n_attr].val.clusterDim.y = 1;
    attr[n_attr].val.clusterDim.z = 1;
    ++n_attr;
  }
  cfg.attrs = attr;
  cfg.numAttrs = n_attr;
  return cudaLaunchKernelEx(&cfg, gemm_sm100_kernel<BN, MODE, PAIR, ROWS>, a.tmA, tmB, a.tmC, p) == cudaSuccess ? 0 : -1;
}

// Tile width, CTA pairing and K slices: the least time by a model of one launch, in us.  What decides is how full the last wave is
// and how wide the tiles that it is paid in: 1,323 rows of gate/up are 192 pair tiles of 256 columns, 2.6 waves of 74 pairs paid
// as three, or 222 of 224 columns, three whole waves; 600 rows are 160 tiles of 256 columns, 1.08 waves paid as two, or 260 of 160,
// the same two waves with five eighths of the columns each (15.5 -> 11.6 us).  So tiles come in the widths of has_width, and
// residual adds may cut them in up to eight K slices.  The model's terms:
//   a k-block of 64: by the rows filled (A box + tile width: L2 -> SM) with a floor, or by a pair's width; up to a sixth less
//   where the launch leaves SMs idle; a wave: 1.08 / 0.77; the last epilogue: by width, the rotary one of 128-column heads dearest;
//   a launch 2.4, a pair 1.25 more.
// Calls of at most 64 rows load activation boxes of 16, 32 or 64 rows: the rest of the MMA's 128 rows is whatever the stage held
// (rows are independent, and rows beyond M go nowhere), where a full box would fill them with zeros at the same cost as data.
// Fitted to 25,000 timings of whole steps in which one projection is given another tile (weights from HBM, the real epilogues:
// decoders 256 to 4,096 wide, heads of 64 and 128, 16 to 8,019 rows): all of a layer's choices together cost 0.5 to 0.7 % of it over the
// best ones (before: 1.4 to 1.8 %; with widths of 64, 128 and 256 and a model by fill rates alone 4 to 5 %).  A fit to launches of
// the plain-store epilogue back to back, their weights in L2, had rated the rotary epilogue of 128-column heads at a fifth (256-wide
// QKV tiles for 128-wide ones, 121 -> 112 us a layer of 2,048 columns at 612 rows) and single tiles against pairs too well
// (gate/up of the same layer 121 -> 117).  Fitted to half of the row counts, the model lost 0.75 % on the others.
// A choice takes ~0.2 us of the host (residual adds 0.5).  It depends on the rows through gemm_row_class alone: a context makes the
// choices of every class when it is created and a call looks its five up.  (Made for every layer of a call they were 1 us of a
// one-layer step's 29 us of enqueueing and 25 us of 24 layers' 430.)
// Tile widths a mode has: whole heads for the rotary epilogues, whole 64-column stores for the plain one; the adds could take any 32
// columns, SwiGLU any 16.  Single CTAs / pairs: adds 64 to 256 without 224 / 96 to 256 (the model would give single CTAs 224 in
// 0.5 % of the problems), SwiGLU 64, 128 to 256 / 128 to 256, plain stores and heads of 64 64, 128, 192, 256 / 128, 192, 256, heads of
// 128 128, 256 / 128, 256, LM head 64, 128, 256 / 128, 256.
constexpr bool has_width(int mode, int bn, bool pair) {
  switch (bn) {
    case 64: return !pair && mode != GS_QKV_ROPE128;
    case 96: return mode == GS_ADD_F32;
    case 160: return mode == GS_ADD_F32 || mode == GS_SWIGLU;
    case 192: return mode == GS_ADD_F32 || mode == GS_SWIGLU || mode == GS_QKV_ROPE || mode == GS_STORE_BF16;
    case 224: return (mode == GS_ADD_F32 && pair) || mode == GS_SWIGLU;
    default: return bn == 128 || bn == 256;
  }
}
// Where 96, 160, 192 or 224 do not divide the output's columns, the last tile reaches beyond: TMA fills weight rows beyond the
// last with zeros (for SwiGLU's gate half they are the first `up` rows instead) and drops columns beyond the output's.
static bool width_fits(int mode, int n_cols, int bn, bool pair) {
  return has_width(mode, bn, pair) && ((bn & (bn - 1)) || n_cols % (mode == GS_SWIGLU ? bn / 2 : bn) == 0);
}
int make_weight_tmaps(WeightMaps* w, const void* base, int rows, int cols, int mode, int* n_made) {
  const int n_cols = mode == GS_SWIGLU ? rows / 2 : rows;
  int bad = 0;
  for (int bn = 64; bn <= 256; bn += 32) {
    if (!width_fits(mode, n_cols, bn, false) && !width_fits(mode, n_cols, bn, true)) continue;
    bad |= make_tmap_2d(&w->half_tile(bn), base, rows, cols, bn / 2);
    ++*n_made;
  }
  return bad;
}
struct TileModel {
  double row, col, least64, least;      // a k-block of a single CTA: a row of the A box, a column, the floor (64 columns wide, wider)
  double pair96, pair0, pair_col;       // of a pair: 96 columns wide, wider
  double alone;                         // what a k-block takes where a launch has one tile
  double wave, wave_pair, pair, cut_col;
};
constexpr TileModel kProjectionModel = {0.00034, 0.00068, 0.117, 0.120, 0.0883, 0.0240, 0.00060, 0.84, 1.08, 0.766, 1.25, 0.00094};
constexpr TileModel kLmHeadModel = {0.00042, 0.00122, 0.150, 0.183, 0.146, 0.0137, 0.00125, 0.75, 0.68, 0.78, 0.9, 0.0};
static TileChoice pick_tile(int mode, int n_cols, int M, int K, int n_sms, int max_splits, bool allow_pair) {
  const int k_blocks = K / KSUB;
  TileChoice best = {mode == GS_QKV_ROPE128 ? 128 : 64, 1, false};
  double best_us = 1e30;
  const TileModel& m = mode == GS_ARGMAX ? kLmHeadModel : kProjectionModel;
  const double epi = mode == GS_ADD_F32 ? 0.00746 : mode == GS_SWIGLU ? 0.0137 : mode == GS_STORE_BF16 ? 0.0036 : mode == GS_ARGMAX ? 0.015 :
                     mode == GS_QKV_ROPE128 ? 0.0314 : 0.0082;   // a column
  for (int pair = allow_pair && M > 64 ? 1 : 0; pair >= 0; --pair) {      // (a pair's tile needs whole boxes)
    for (int bn = 256; bn >= 64; bn -= 32) {
      if (!width_fits(mode, n_cols, bn, pair != 0)) continue;
      const int out_n = (mode == GS_SWIGLU) ? bn / 2 : bn;
      const int tile_m = pair ? 2 * BM : BM;
      const int walkers = pair ? n_sms / 2 : n_sms;
      const long long tiles = (long long)((M + tile_m - 1) / tile_m) * ((n_cols + out_n - 1) / out_n);
      const double fill = m.row * gemm_a_box_rows(M) + m.col * bn, least = bn == 64 ? m.least64 : m.least;
      double kb_us = pair ? (bn <= 96 ? m.pair96 : m.pair0 + m.pair_col * bn) : (fill > least ? fill : least);
      // The LM head's weights come from HBM.  One row tile of it waits for them, and has more of them under way on narrower tiles:
      // at 1 to 128 rows 128 columns take 0.91 to 1.00 of 256 columns' time (vocabularies of 32,768 to 131,072, K of 512 to 4,096,
      // L2 flushed; 16 rows, 131,072 x 2,048: 107 and 114 us with the call's two small kernels).  Beyond, a pair takes a tile of
      // weights once for 256 rows (144 rows: 20.3 us on 256-wide tiles, 17.9 on pairs of that width): 1.11 fits 360 timings at 1 to
      // 2,049 rows, with choices 2.0 % off the best on average; 1.15 put 640 rows of large vocabularies on pairs, up to 14 % slower.
      if (mode == GS_ARGMAX && !pair && M <= BM && bn == 256) continue;
      if (mode == GS_ARGMAX && !pair && M > BM) kb_us *= 1.11;
      for (int sp = 1; sp <= max_splits; ++sp) {
        const int kbs = (k_blocks + sp - 1) / sp;
        if (sp > 1 && (kbs < 2 || (long long)(sp - 1) * kbs >= k_blocks)) continue;
        const long long units = tiles * sp;
        const long long rounds = (units + walkers - 1) / walkers;
        const double load = units < walkers ? (double)units / walkers : 1.0;
        const double us = 2.4 + (pair ? m.pair : 0.0) + rounds * (kbs * kb_us * (m.alone + (1.0 - m.alone) * load) + (pair ? m.wave_pair : m.wave)) +
                          epi * bn + (sp > 1 ? m.cut_col * bn : 0.0);
        if (us < 0.99 * best_us) { best_us = us; best = {bn, sp, pair != 0}; }      // (as good: the wider one, with less traffic)
      }
    }
  }
  return best;
}

template <int MODE, bool PAIR, int BN = 64>
static int launch_width(cudaStream_t st, const GemmSm100Args& a, int bn, int splits) {
  if constexpr (has_width(MODE, BN, PAIR)) {
    if (bn == BN) {
      if constexpr (BN == 64) {
        if (a.M <= 16) return launch_one<BN, MODE, PAIR, 16>(st, a, splits);
        if (a.M <= 64) return launch_one<BN, MODE, PAIR, 64>(st, a, splits);
      }
      return launch_one<BN, MODE, PAIR>(st, a, splits);
    }
  }
  if constexpr (BN < 256) return launch_width<MODE, PAIR, BN + 32>(st, a, bn, splits);
  return -1;
}

// The shared memory each kernel is launched with.  Asked for when a context is created, which also loads the kernels, ~50 us each:
// the first step that picks a width does not wait for that.  A context loads the modes that its model's steps have, 43 kernels
// with heads of 64 and 38 with heads of 128, of 56; the plain store is hsd_op_linear's alone.
template <int BN, int MODE, bool PAIR, int ROWS = BM>
static bool allow_smem_one() {
  return cudaFuncSetAttribute(gemm_sm100_kernel<BN, MODE, PAIR, ROWS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              Cfg<BN, PAIR, ROWS>::SMEM_BYTES) == cudaSuccess;
}
template <int MODE, bool PAIR, int BN = 64>
static bool allow_smem() {
  bool ok = true;
  if constexpr (has_width(MODE, BN, PAIR)) ok = allow_smem_one<BN, MODE, PAIR>();
  if constexpr (has_width(MODE, BN, PAIR) && BN == 64) ok = allow_smem_one<BN, MODE, PAIR, 16>() && allow_smem_one<BN, MODE, PAIR, 64>() && ok;
  if constexpr (BN < 256) ok = allow_smem<MODE, PAIR, BN + 32>() && ok;
  return ok;
}
template <int MODE>
static int prepare_mode(int device, int* n_kernels) {
  static std::atomic<bool> done[kMaxDevices];      // the attribute is per device; contexts may be created by several threads
  for (int bn = 64; bn <= 256; bn += 32)
    *n_kernels += has_width(MODE, bn, false) * (bn == 64 ? 3 : 1) + has_width(MODE, bn, true);
  if (!done[device]) {
    if (!allow_smem<MODE, false>() || !allow_smem<MODE, true>()) return -1;
    done[device] = true;
  }
  return 0;
}
int gemm_sm100_prepare(int mode, int* n_kernels) {
  int device = -1;
  if (cudaGetDevice(&device) != cudaSuccess || device < 0 || device >= kMaxDevices) return -1;
  switch (mode) {
    case GS_STORE_BF16: return prepare_mode<GS_STORE_BF16>(device, n_kernels);
    case GS_ADD_F32: return prepare_mode<GS_ADD_F32>(device, n_kernels);
    case GS_SWIGLU: return prepare_mode<GS_SWIGLU>(device, n_kernels);
    case GS_ARGMAX: return prepare_mode<GS_ARGMAX>(device, n_kernels);
    case GS_QKV_ROPE: return prepare_mode<GS_QKV_ROPE>(device, n_kernels);
    case GS_QKV_ROPE128: return prepare_mode<GS_QKV_ROPE128>(device, n_kernels);
    default: return -1;
  }
}

TileChoice gemm_choose_tile(const GemmSm100Args& a, int force_bn, int force_splits) {
  const int n_cols = (a.mode == GS_SWIGLU) ? a.n_out / 2 : a.n_out;
  const TileChoice none = {0, 0, false};
  TileChoice c = pick_tile(a.mode, n_cols, gemm_class_rows(gemm_row_class(a.M)), a.K, a.n_sms, (a.mode == GS_ADD_F32 && a.max_splits > 1) ? a.max_splits : 1, a.pair != 0);
  if (force_bn) {
    c.pair = force_bn > 256;                                // a CTA pair on tiles of 256 rows and 256 columns less
    c.bn = c.pair ? force_bn - 256 : force_bn;
    if (!width_fits(a.mode, n_cols, c.bn, c.pair)) return none;
    if (c.pair && a.M <= 64) {                              // a pair's tile needs whole boxes: one CTA in its place,
      c.pair = false;                                       // of 256 columns where only pairs have the width
      if (!has_width(a.mode, c.bn, false)) c.bn = 256;
      if (!width_fits(a.mode, n_cols, c.bn, false)) return none;
    }
  }
  if (force_splits) {
    const int kbs = (a.K / KSUB + force_splits - 1) / force_splits;
    if (a.mode != GS_ADD_F32 || (force_splits - 1) * kbs >= a.K / KSUB) return none;
    c.splits = force_splits;
  }
  return c;
}

template <int MODE>
static int launch_mode(cudaStream_t st, const GemmSm100Args& a) {
  return a.tile.pair ? launch_width<MODE, true>(st, a, a.tile.bn, a.tile.splits) : launch_width<MODE, false>(st, a, a.tile.bn, a.tile.splits);
}

int launch_gemm_sm100(cudaStream_t st, const GemmSm100Args& a) {
  if (a.M <= 0) return 0;
  if (a.K % KSUB || a.n_out % 64 || !a.tmB) return -1;
  switch (a.mode) {
    case GS_STORE_BF16: return launch_mode<GS_STORE_BF16>(st, a);
    case GS_ADD_F32: return launch_mode<GS_ADD_F32>(st, a);
    case GS_SWIGLU: return launch_mode<GS_SWIGLU>(st, a);
    case GS_ARGMAX: return launch_mode<GS_ARGMAX>(st, a);
    case GS_QKV_ROPE: return launch_mode<GS_QKV_ROPE>(st, a);
    case GS_QKV_ROPE128: return launch_mode<GS_QKV_ROPE128>(st, a);
    default: return -1;
  }
}

}  // namespace hsd
