// Memory- and latency-bound kernels of the verify step: row metadata + checks, embedding gather,
// RMSNorm, RoPE + paged KV write, the plain SIMT attention (debug cross-check), accept/emit, KV commit.
#include "hsd_attn_plan.cuh"
#include "hsd_kernels.h"

namespace hsd {

const char* kernel_class_name(int kc) {
  static const char* names[KC_COUNT] = {"setup_rows", "rmsnorm",   "gemm_qkv",       "rope_kv_write", "attention", "gemm_o",
                                        "gemm_gate_up", "gemm_down", "lm_head_argmax", "accept_emit",   "kv_commit", "debug"};
  return (kc >= 0 && kc < KC_COUNT) ? names[kc] : "?";
}

// ------------------------------------------------------------------------------------------------
// Row metadata, embedding gather and the LM head's cleared rows: what a step needs before its first layer, in one launch.
// A CTA takes kSetupRows packed rows whatever the sequences they belong to; the first CTA writes the per-sequence metadata
// and makes the attention plan from it, beside the others' work.
// Validates what the host cannot see (device-resident offsets, lengths and tables).  A CTA leaves its verdict {code, index}
// in `verdict`, and the kernel that follows (the first RMSNorm) turns the verdicts into the status words: nothing has to be zeroed first.  Every kernel that follows an indirection returns early
// on a violation.
// (Separate launches for the status words, the metadata by sequence, the gather and the cleared rows, with the parent
// walk through global memory, took 16 to 30 us of a step.  The plan in a launch of its own behind this one: one small layer
// 53 us, now 50; 16 plain rows 0.8925 ms, now 0.8895; one lane's 128-node tree 1.186 ms, now 1.180.)
constexpr int kSetupThreads = 256, kSetupMaxCu = 1024;
__device__ __forceinline__ int setup_cu(const SetupArgs& a, int s) { return a.cu_q ? a.cu_q[s] : (s ? a.total_q : 0); }

__global__ void __launch_bounds__(kSetupThreads) setup_rows_kernel(SetupArgs a, KvView kv, RowMeta rm) {
  // rotary frequency base^(-2f/D) of this thread (half divides the CTA: a thread stays with one), in double so that the
  // angles of long contexts keep accuracy
  const int half = a.head_dim / 2, f = threadIdx.x % half;
  const double inv = exp2(-(double)(2 * f) / (double)a.head_dim * log2((double)a.rope_base));
  pdl_wait();               // everything below reads or writes what earlier kernels of the stream produced
  pdl_launch_dependents();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  __shared__ int s_cu[kSetupMaxCu + 1];
  __shared__ int s_code, s_where;
  __shared__ int s_par[HSD_MAX_TREE_ROWS + kSetupRows];
  __shared__ int s_tok[kSetupRows], s_len[kSetupRows];
  __shared__ int s_warp[kSetupThreads / 32];
  int2* verdict = a.verdict + (blockIdx.x ? blockIdx.x - 1 : gridDim.x - 1);     // the rows' ahead of the sequences'
  if (tid == 0) s_code = s_where = 0;
  __syncthreads();
  auto fail = [&](int code, int where) {
    if (atomicCAS(&s_code, 0, code) == 0) s_where = where;
  };
  // every CTA checks the offsets once, and keeps them where they fit
  int bad = 0;
  for (int s = tid; s < a.n_seqs; s += kSetupThreads) {
    const int lo = setup_cu(a, s), n = setup_cu(a, s + 1) - lo;
    if (n < 0) bad = DEV_CU_Q;
    if (n > a.max_q_len && !bad) bad = DEV_TOO_LONG;
    if (s < kSetupMaxCu) s_cu[s] = lo;
  }
  if (tid == 0 && (setup_cu(a, 0) != 0 || setup_cu(a, a.n_seqs) != a.total_q)) bad = DEV_CU_Q;
  if (bad) atomicMax(&s_code, bad == DEV_TOO_LONG ? 2 : 1);
  __syncthreads();
  if (s_code) {
    if (tid == 0) *verdict = make_int2(s_code == 2 ? DEV_TOO_LONG : DEV_CU_Q, 0);
    return;
  }

  if (blockIdx.x == 0) {                    // the sequences, with the exclusive scan of their attention q-tiles
    int base = 0;
    for (int s0 = 0; s0 < a.n_seqs; s0 += kSetupThreads) {
      const int s = s0 + tid;
      int q0 = 0, n = 0, slot = 0, L = 0;
      if (s < a.n_seqs) {
        q0 = setup_cu(a, s);
        n = setup_cu(a, s + 1) - q0;
        slot = a.seq_slots ? a.seq_slots[s] : a.slot_base + s;
        if (slot < 0 || slot >= kv.n_slots) {
          fail(DEV_KV_CAPACITY, s);
        } else {
          L = kv.seq_lens[slot];
          if (L < 0 || (long long)L + n > (long long)kv.max_blocks * HSD_KV_BLOCK) fail(DEV_KV_CAPACITY, s);
        }
      }
      const int tiles = (n + a.tokens_per_tile - 1) / a.tokens_per_tile;
      int incl = tiles;
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
      }
      if (lane == 31) s_warp[warp] = incl;
      __syncthreads();
      int before = base, all = 0;
      for (int w = 0; w < kSetupThreads / 32; ++w) {
        if (w < warp) before += s_warp[w];
        all += s_warp[w];
      }
      if (s < a.n_seqs) {
        rm.seq_q0[s] = q0;
        rm.seq_n[s] = n;
        rm.seq_len[s] = L;
        rm.seq_slot[s] = slot;
        rm.seq_tile0[s] = before + incl - tiles;
      }
      base += all;
      __syncthreads();
    }
    for (int r = a.total_q + tid; r < a.n_seqs; r += kSetupThreads) a.row_best[r] = 0ull;   // (LM-head rows of empty sequences)
    if (tid == 0) {
      rm.seq_tile0[a.n_seqs] = base;
      *verdict = make_int2(s_code, s_where);
    }
    __syncthreads();
    if (a.make_plan && !s_code) make_attn_plan<kSetupThreads>(rm, a.plan, kv, a.rule, a.n_seqs, base, a.tokens_per_tile);
    return;
  }

  const int r0 = (blockIdx.x - 1) * kSetupRows, n_rows = min(kSetupRows, a.total_q - r0);
  const int par0 = max(0, r0 - HSD_MAX_TREE_ROWS);      // a row's ancestors lie among the 127 packed rows before it
  if (a.parent)
    for (int j = par0 + tid; j < r0 + n_rows; j += kSetupThreads) s_par[j - par0] = a.parent[j];
  __syncthreads();
  if (tid < n_rows) {
    const int r = r0 + tid;
    int lo = 0, hi = a.n_seqs;                          // the sequence of row r: the last that begins at or before it
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if ((mid < kSetupMaxCu ? s_cu[mid] : setup_cu(a, mid)) <= r) lo = mid; else hi = mid;
    }
    const int i = lo, q0 = lo < kSetupMaxCu ? s_cu[lo] : setup_cu(a, lo);
    const int j = r - q0, n = setup_cu(a, i + 1) - q0;
    int tok, nxt = -1;
    if (a.tokens) {
      tok = a.tokens[r];
      if (j + 1 < n) nxt = a.tokens[r + 1];
    } else {
      tok = (j == 0) ? a.pending[0] : a.draft[j - 1];
      if (j + 1 < n) nxt = a.draft[j];
    }
    const int slot = a.seq_slots ? a.seq_slots[i] : a.slot_base + i;
    int L = 0, phys = 0;
    if (slot < 0 || slot >= kv.n_slots) {
      fail(DEV_KV_CAPACITY, i);
    } else {
      L = kv.seq_lens[slot];
      if (L < 0 || (long long)L + n > (long long)kv.max_blocks * HSD_KV_BLOCK) {
        fail(DEV_KV_CAPACITY, i);
        L = 0;
      } else {
        phys = kv.block_table[(size_t)slot * kv.max_blocks + (L + j) / HSD_KV_BLOCK];
        if (phys < 0 || phys >= kv.n_blocks) {
          fail(DEV_BLOCK_RANGE, r);
          phys = 0;
        }
      }
    }
    if (tok >= a.vocab || (tok < 0 && !a.allow_embed_rows)) {
      fail(DEV_TOKEN_RANGE, r);
      tok = 0;
    }
    if (tok < 0) tok = -1;
    // Candidate tree: a row's rotary position is its depth below the pending token, not its index in the call
    // (Sec. 3.2: a node continues the path pi(v), whatever else is packed beside it).
    int d = 0;
    if (a.parent) {
      uint32_t m[4] = {0u, 0u, 0u, 0u};
      const int own = s_par[r - par0];
      int pj = j;
      bool ok = j < HSD_MAX_TREE_ROWS;
      if (ok) m[j >> 5] |= 1u << (j & 31);
      if (j > 0 && own == -2) pj = 0;                   // padding row: no parent, no children, sees only itself
      while (ok && pj > 0) {
        const int pp = s_par[q0 + pj - par0];
        if (pp < 0 || pp >= pj) { ok = false; break; }
        pj = pp;
        m[pj >> 5] |= 1u << (pj & 31);
        ++d;
      }
      if (j == 0 && own != -1) ok = false;
      if (!ok) {
        fail(DEV_TREE, r);
        d = 0;
      }
      rm.anc[r] = make_uint4(m[0], m[1], m[2], m[3]);
      const bool child = ok && j > 0 && own >= 0;
      rm.child_src[r] = child ? q0 + own : r;
      rm.child_tok[r] = child ? tok : -1;
    }
    rm.row_seq[r] = i;
    rm.row_pos[r] = L + (a.parent ? d : j);
    rm.row_tok[r] = tok;
    rm.row_kv[r] = phys * HSD_KV_BLOCK + (L + j) % HSD_KV_BLOCK;
    rm.row_next[r] = (a.allow_embed_rows || a.parent) ? -1 : nxt;
    a.row_best[r] = 0ull;                               // the LM head's running best and captured logit
    a.zdraft[r] = __int_as_float(0x7fc00000);
    s_tok[tid] = tok;
    s_len[tid] = L + (a.parent ? d : j);
  }
  __syncthreads();
  if (tid == 0) *verdict = make_int2(s_code, s_where);
  // embedding gather: x[r] = fp32(table[tok]) or fp32(embeds[r]), a warp per row, 16-byte loads
  for (int k = warp; k < n_rows; k += kSetupThreads / 32) {
    const int tok = s_tok[k];
    const bf16* src = tok >= 0 ? a.table + (size_t)tok * a.d : a.embeds + (size_t)(r0 + k) * a.d;
    float* dst = a.x + (size_t)(r0 + k) * a.d;
#pragma unroll 4
    for (int c = lane * 8; c < a.d; c += 256) {
      const uint4 v = *reinterpret_cast<const uint4*>(src + c);
      *reinterpret_cast<float4*>(dst + c) = make_float4(bf16_lo(v.x), bf16_hi(v.x), bf16_lo(v.y), bf16_hi(v.y));
      *reinterpret_cast<float4*>(dst + c + 4) = make_float4(bf16_lo(v.z), bf16_hi(v.z), bf16_lo(v.w), bf16_hi(v.w));
    }
  }
  // rotary table: (cos, sin) of the position times the frequency
  for (int k = tid / half; k < n_rows; k += kSetupThreads / half) {
    double sn, cs;
    sincos((double)s_len[k] * inv, &sn, &cs);
    rm.rope_cs[(size_t)(r0 + k) * half + f] = make_float2((float)cs, (float)sn);
  }
}

int setup_ctas(int total_q) { return (total_q + kSetupRows - 1) / kSetupRows + 1; }
void launch_setup_rows(cudaStream_t st, const SetupArgs& a, const KvView& kv, const RowMeta& rm, bool pdl) {
  launch_kernel(setup_rows_kernel, dim3(setup_ctas(a.total_q)), dim3(kSetupThreads), 0, st, pdl, a, kv, rm);
}

// ------------------------------------------------------------------------------------------------
// RMSNorm: h = bf16(x * rsqrt(mean(x^2) + eps) * gain).  One warp per row; the row stays in registers
// between the reduction and the scaling (d <= 4096), so x is read once.
template <int VEC>   // VEC float4 per lane: d = 128 * VEC
__global__ void rmsnorm_kernel(const float* __restrict__ x, const bf16* __restrict__ gain, bf16* __restrict__ h,
                               int rows, int d, float eps, const int* __restrict__ sel_rows, int src_rows,
                               const int* __restrict__ status, const int2* verdict, int n_verdicts, int* status_out) {
  pdl_wait();               // everything below reads or writes what earlier kernels of the step produced
  pdl_launch_dependents();
  if (verdict && blockIdx.x == gridDim.x - 1) {        // one CTA more: the status words of the step
    status_from_verdicts(verdict, n_verdicts, status_out);
    return;
  }
  const int r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (r >= rows) return;
  const int lane = threadIdx.x & 31;
  // the gather form follows an index an earlier kernel of the step wrote: after a failed device-side check that
  // index was never written, so nothing is read through it (and an index outside the source is never followed)
  if (sel_rows && status && *status) return;
  const int src = sel_rows ? sel_rows[r] : r;
  if (src < 0 || src >= src_rows) return;
  const float4* xp = reinterpret_cast<const float4*>(x + (size_t)src * d);
  const uint2* gp = reinterpret_cast<const uint2*>(gain);
  float4 v[VEC];
  uint2 gv[VEC];
#pragma unroll
  for (int i = 0; i < VEC; ++i) v[i] = xp[lane + 32 * i];
#pragma unroll
  for (int i = 0; i < VEC; ++i) gv[i] = __ldg(gp + lane + 32 * i);      // in flight together with the row
  float ss = 0.f;
#pragma unroll
  for (int i = 0; i < VEC; ++i) ss += v[i].x * v[i].x + v[i].y * v[i].y + v[i].z * v[i].z + v[i].w * v[i].w;
  for (int o = 16; o; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  const float rs = rsqrtf(ss / (float)d + eps);
  uint2* hp = reinterpret_cast<uint2*>(h + (size_t)r * d);
#pragma unroll
  for (int i = 0; i < VEC; ++i) {
    const uint2 g = gv[i];
    uint2 o;
    o.x = pack_bf16(v[i].x * rs * bf16_lo(g.x), v[i].y * rs * bf16_hi(g.x));
    o.y = pack_bf16(v[i].z * rs * bf16_lo(g.y), v[i].w * rs * bf16_hi(g.y));
    hp[lane + 32 * i] = o;
  }
}
static void launch_rmsnorm_any(cudaStream_t st, const float* x, const bf16* gain, bf16* h, int rows, int d, float eps,
                               const int* sel_rows, int src_rows, const int* status, const int2* verdict, int n_verdicts,
                               int* status_out, int n_sms, bool pdl) {
  // Four rows a CTA while no SM gets two of the launch's CTAs by that, eight otherwise: 16 rows 1.95 us a launch with eight and 1.81
  // with four, 513 rows 2.55 and 2.37, ~1,090 rows 3.19 and 3.74 (two rows a CTA as four, sixteen 2.57 / 2.78 / 3.25).
  const int per = (rows + 3) / 4 + (verdict ? 1 : 0) <= n_sms ? 4 : 8;
  dim3 grid((rows + per - 1) / per + (verdict ? 1 : 0)), block(32 * per);
#define HSD_RMS_CASE(V)                                                                                                  \
  case V:                                                                                                                \
    launch_kernel(rmsnorm_kernel<V>, grid, block, 0, st, pdl, x, gain, h, rows, d, eps, sel_rows, src_rows, status, verdict, \
                  n_verdicts, status_out);                                                                               \
    break;
  switch (d / 128) {
    HSD_RMS_CASE(1) HSD_RMS_CASE(2) HSD_RMS_CASE(4) HSD_RMS_CASE(8) HSD_RMS_CASE(16) HSD_RMS_CASE(32)
    default: break;   // hsd_create rejects other widths
  }
#undef HSD_RMS_CASE
}
void launch_rmsnorm(cudaStream_t st, const float* x, const bf16* gain, bf16* h, int rows, int d, float eps,
                    const int* sel_rows, int src_rows, const int* status, int n_sms, bool pdl) {
  if (rows > 0) launch_rmsnorm_any(st, x, gain, h, rows, d, eps, sel_rows, src_rows, status, nullptr, 0, nullptr, n_sms, pdl);
}
void launch_first_rmsnorm(cudaStream_t st, const float* x, const bf16* gain, bf16* h, int rows, int d, float eps,
                          const int2* verdict, int n_verdicts, int* status, int n_sms, bool pdl) {
  launch_rmsnorm_any(st, x, gain, h, rows, d, eps, nullptr, rows, nullptr, verdict, n_verdicts, status, n_sms, pdl);
}

// The final norm of a tree step: h as above, and for every node the logit of its own token under its PARENT's distribution,
// which the traversal compares (Eq. 10): the parent's normed row, made again from x and rounded as it is in h, times the
// token's row of the LM head.  A warp per row; bound by the latency of the token's row (2 KB at d = 1024, scattered in HBM).
// (As rows T .. 2T of the LM head's own GEMM, each against the whole vocabulary for one captured column, 2,048 nodes took
// 162 us there and 4.5 us in the norm; now 78 and 6.  128 nodes: 18 and 2, now 14 and 4.7.)
template <int VEC>
__global__ void tree_final_norm_kernel(const float* __restrict__ x, const bf16* __restrict__ gain, bf16* __restrict__ h, int rows, int d,
                                       float eps, const int* __restrict__ child_src, const int* __restrict__ child_tok,
                                       const bf16* __restrict__ lm_head, int vocab, float* __restrict__ zchild,
                                       const int* __restrict__ status) {
  // The indices come from the step's set-up, which the kernel before this one waited for before it let this one start: they and
  // the token's row are under way while that kernel still runs.
  const int r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  const bool dead = r >= rows || __ldcg(status);         // (after a failed device-side check the indices were never written)
  const int src = dead ? -1 : __ldcg(child_src + r), tok = dead ? -1 : __ldcg(child_tok + r);
  const bool child = tok >= 0 && tok < vocab && src >= 0 && src < rows;
  const uint2* gp = reinterpret_cast<const uint2*>(gain);
  uint2 w[VEC], o[VEC];
  if (child) {
    const uint2* wp = reinterpret_cast<const uint2*>(lm_head + (size_t)tok * d);
#pragma unroll
    for (int i = 0; i < VEC; ++i) w[i] = __ldg(wp + lane + 32 * i);
  }
  pdl_wait();               // x is what the kernel before wrote
  pdl_launch_dependents();
  if (dead) return;
  auto normed = [&](int row) {
    const float4* xp = reinterpret_cast<const float4*>(x + (size_t)row * d);
    float4 v[VEC];
#pragma unroll
    for (int i = 0; i < VEC; ++i) v[i] = xp[lane + 32 * i];
    float ss = 0.f;
#pragma unroll
    for (int i = 0; i < VEC; ++i) ss += v[i].x * v[i].x + v[i].y * v[i].y + v[i].z * v[i].z + v[i].w * v[i].w;
    for (int s = 16; s; s >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, s);
    const float rs = rsqrtf(ss / (float)d + eps);
#pragma unroll
    for (int i = 0; i < VEC; ++i) {
      const uint2 g = __ldg(gp + lane + 32 * i);
      o[i] = make_uint2(pack_bf16(v[i].x * rs * bf16_lo(g.x), v[i].y * rs * bf16_hi(g.x)),
                        pack_bf16(v[i].z * rs * bf16_lo(g.y), v[i].w * rs * bf16_hi(g.y)));
    }
  };
  normed(r);
  uint2* hp = reinterpret_cast<uint2*>(h + (size_t)r * d);
#pragma unroll
  for (int i = 0; i < VEC; ++i) hp[lane + 32 * i] = o[i];
  if (!child) return;
  normed(src);
  float z = 0.f;
#pragma unroll
  for (int i = 0; i < VEC; ++i)
    z += (bf16_lo(o[i].x) * bf16_lo(w[i].x) + bf16_hi(o[i].x) * bf16_hi(w[i].x)) +
         (bf16_lo(o[i].y) * bf16_lo(w[i].y) + bf16_hi(o[i].y) * bf16_hi(w[i].y));
  for (int s = 16; s; s >>= 1) z += __shfl_xor_sync(0xffffffffu, z, s);
  if (lane == 0) zchild[r] = z;
}
void launch_tree_final_norm(cudaStream_t st, const float* x, const bf16* gain, bf16* h, int rows, int d, float eps,
                            const RowMeta& rm, const bf16* lm_head, int vocab, float* zchild, const int* status, bool pdl) {
#define HSD_TREE_NORM_CASE(V)                                                                                                   \
  case V:                                                                                                                      \
    launch_kernel(tree_final_norm_kernel<V>, dim3((rows + 7) / 8), dim3(256), 0, st, pdl, x, gain, h, rows, d, eps, rm.child_src, \
                  rm.child_tok, lm_head, vocab, zchild, status);                                                               \
    break;
  switch (d / 128) {
    HSD_TREE_NORM_CASE(1) HSD_TREE_NORM_CASE(2) HSD_TREE_NORM_CASE(4) HSD_TREE_NORM_CASE(8) HSD_TREE_NORM_CASE(16) HSD_TREE_NORM_CASE(32)
    default: break;   // hsd_create rejects other widths
  }
#undef HSD_TREE_NORM_CASE
}

__global__ void select_last_rows_kernel(RowMeta rm, int n_seqs, int* sel_rows, const int* status) {
  pdl_wait();               // everything below reads or writes what earlier kernels of the step produced
  pdl_launch_dependents();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_seqs) return;
  // after a failed check the per-sequence metadata was not written: name no row at all
  sel_rows[i] = *status ? -1 : rm.seq_q0[i] + max(rm.seq_n[i], 1) - 1;
}
void launch_select_last_rows(cudaStream_t st, const RowMeta& rm, int n_seqs, int* sel_rows, const int* status, bool pdl) {
  launch_kernel(select_last_rows_kernel, dim3((n_seqs + 127) / 128), dim3(128), 0, st, pdl, rm, n_seqs, sel_rows, status);
}

__global__ void clear_best_kernel(unsigned long long* row_best, float* zdraft, int rows) {
  pdl_wait();               // everything below reads or writes what earlier kernels of the step produced
  pdl_launch_dependents();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < rows) {
    row_best[i] = 0ull;
    if (zdraft) zdraft[i] = __int_as_float(0x7fc00000);
  }
}
void launch_clear_best(cudaStream_t st, unsigned long long* row_best, float* zdraft, int rows, bool pdl) {
  launch_kernel(clear_best_kernel, dim3((rows + 255) / 256), dim3(256), 0, st, pdl, row_best, zdraft, rows);
}

__global__ void unpack_best_kernel(const unsigned long long* row_best, int rows, int* argmax, float* zmax) {
  pdl_wait();               // everything below reads or writes what earlier kernels of the step produced
  pdl_launch_dependents();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < rows) {
    const unsigned long long b = row_best[i];
    if (argmax) argmax[i] = key_col(b);
    if (zmax) zmax[i] = key_value(b);
  }
}
void launch_unpack_best(cudaStream_t st, const unsigned long long* row_best, int rows, int* argmax, float* zmax,
                        bool pdl) {
  launch_kernel(unpack_best_kernel, dim3((rows + 255) / 256), dim3(256), 0, st, pdl, row_best, rows, argmax, zmax);
}

// ------------------------------------------------------------------------------------------------
// RoPE + paged KV write from an fp32 qkv row (SIMT path; the tensor-core path fuses this into the
// QKV projection's epilogue).  One warp per (row, head); lane i holds dims i and i + 32.
__global__ void rope_kvwrite_kernel(const float* __restrict__ qkv, RowMeta rm, KvView kv, ModelDims md, int layer,
                                    bf16* __restrict__ q, int T, const int* status, const bf16* __restrict__ q_norm,
                                    const bf16* __restrict__ k_norm) {
  if (*status) return;
  const int heads = md.Hq + 2 * md.Hkv;
  const int w = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (w >= T * heads) return;
  const int r = w / heads, hd = w % heads, lane = threadIdx.x & 31;
  const float* src = qkv + (size_t)r * md.qkv_out + hd * 64;
  float a = src[lane], b = src[lane + 32];
  const int phys = rm.row_kv[r];
  const size_t blk_base = ((size_t)layer * kv.n_blocks + phys / 64) * md.Hkv;
  const int off = phys % 64;
  if (hd < md.Hq + md.Hkv) {
    if (q_norm) {       // per-head RMSNorm over the 64 dims before the rotation
      float ss = a * a + b * b;
      for (int o = 16; o; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
      const float rs = rsqrtf(ss * (1.f / 64.f) + md.eps);
      const bf16* g = hd < md.Hq ? q_norm : k_norm;
      a *= rs * __bfloat162float(g[lane]);
      b *= rs * __bfloat162float(g[lane + 32]);
    }
    const float2 cs = rm.rope_cs[(size_t)r * 32 + lane];
    const float ra = a * cs.x - b * cs.y, rb = b * cs.x + a * cs.y;
    if (hd < md.Hq) {
      bf16* dst = q + (size_t)r * md.Hq * 64 + hd * 64;
      dst[lane] = __float2bfloat16(ra);
      dst[lane + 32] = __float2bfloat16(rb);
    } else {
      bf16* dst = kv.k_pool + ((blk_base + (hd - md.Hq)) * 64 + off) * 64;
      dst[lane] = __float2bfloat16(ra);
      dst[lane + 32] = __float2bfloat16(rb);
    }
  } else {
    bf16* dst = kv.v_pool + ((blk_base + (hd - md.Hq - md.Hkv)) * 64 + off) * 64;
    dst[lane] = __float2bfloat16(a);
    dst[lane + 32] = __float2bfloat16(b);
  }
}
void launch_rope_kvwrite(cudaStream_t st, const float* qkv, const RowMeta& rm, const KvView& kv, const ModelDims& md,
                         int layer, bf16* q, int T, const int* status, const bf16* q_norm, const bf16* k_norm) {
  const long long warps = (long long)T * (md.Hq + 2 * md.Hkv);
  rope_kvwrite_kernel<<<(unsigned)((warps + 7) / 8), 256, 0, st>>>(qkv, rm, kv, md, layer, q, T, status, q_norm, k_norm);
}

// ------------------------------------------------------------------------------------------------
// Plain SIMT attention (debug cross-check): one warp per (row, q head), online softmax over 32-key chunks.
__global__ void attn_simt_kernel(const bf16* __restrict__ q, RowMeta rm, KvView kv, ModelDims md, int layer,
                                 bf16* __restrict__ out, int T, const int* status) {
  if (*status) return;
  const int w = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (w >= T * md.Hq) return;
  const int r = w / md.Hq, hq = w % md.Hq, lane = threadIdx.x & 31;
  const int kvh = hq / md.group;
  const int seq = rm.row_seq[r];
  const int slot = rm.seq_slot[seq];
  const int n_keys = rm.row_pos[r] + 1;            // keys at positions 0 .. pos (causal, own row included)
  __shared__ float s_q[8][64];
  float* qs = s_q[threadIdx.x >> 5];
  const bf16* qp = q + (size_t)r * md.Hq * 64 + hq * 64;
  qs[lane] = __bfloat162float(qp[lane]) * 0.125f;   // 1/sqrt(64)
  qs[lane + 32] = __bfloat162float(qp[lane + 32]) * 0.125f;
  __syncwarp();
  float m = -INFINITY, l = 0.f, o0 = 0.f, o1 = 0.f;
  const int* bt = kv.block_table + (size_t)slot * kv.max_blocks;
  for (int k0 = 0; k0 < n_keys; k0 += 32) {
    const int key = k0 + lane;
    const int phys = bt[k0 / 64];                   // a 32-key chunk never straddles a 64-token block
    const size_t tile = ((size_t)layer * kv.n_blocks + phys) * md.Hkv + kvh;
    float s = -INFINITY;
    if (key < n_keys) {
      const uint4* kp = reinterpret_cast<const uint4*>(kv.k_pool + (tile * 64 + key % 64) * 64);
      float acc = 0.f;
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        uint4 v = kp[c];
        const float* qq = qs + c * 8;
        acc += qq[0] * bf16_lo(v.x) + qq[1] * bf16_hi(v.x) + qq[2] * bf16_lo(v.y) + qq[3] * bf16_hi(v.y) +
               qq[4] * bf16_lo(v.z) + qq[5] * bf16_hi(v.z) + qq[6] * bf16_lo(v.w) + qq[7] * bf16_hi(v.w);
      }
      s = acc;
    }
    float cm = s;
    for (int o = 16; o; o >>= 1) cm = fmaxf(cm, __shfl_xor_sync(0xffffffffu, cm, o));
    const float m_new = fmaxf(m, cm);
    const float p = (key < n_keys) ? __expf(s - m_new) : 0.f;
    float ps = p;
    for (int o = 16; o; o >>= 1) ps += __shfl_xor_sync(0xffffffffu, ps, o);
    const float scale = __expf(m - m_new);
    l = l * scale + ps;
    o0 *= scale;
    o1 *= scale;
    m = m_new;
    // V tile [tok][dim]: lane owns dims lane and lane + 32
    const bf16* vt = kv.v_pool + tile * 4096;
    const int tok0 = k0 % 64;
    const int cnt = min(32, n_keys - k0);
    for (int t = 0; t < cnt; ++t) {
      const float pt = __shfl_sync(0xffffffffu, p, t);
      o0 += pt * __bfloat162float(vt[(size_t)(tok0 + t) * 64 + lane]);
      o1 += pt * __bfloat162float(vt[(size_t)(tok0 + t) * 64 + lane + 32]);
    }
  }
  bf16* op = out + (size_t)r * md.Hq * 64 + hq * 64;
  op[lane] = __float2bfloat16(o0 / l);
  op[lane + 32] = __float2bfloat16(o1 / l);
}
void launch_attn_simt(cudaStream_t st, const bf16* q, const RowMeta& rm, const KvView& kv, const ModelDims& md,
                      int layer, bf16* out, int T, const int* status) {
  const long long warps = (long long)T * md.Hq;
  attn_simt_kernel<<<(unsigned)((warps + 7) / 8), 256, 0, st>>>(q, rm, kv, md, layer, out, T, status);
}

// ------------------------------------------------------------------------------------------------
// Draft compare + longest-prefix accept + emit.  One CTA per sequence: a warp per sequence spent 45 us on a 2,049-row chunk,
// two dependent reads for every 32 rows.
// Row j (0-based) of a sequence holds the distribution after [.., pending, d_1..d_j]; its next draft token is
// d_{j+1}.  a = first j < k whose test fails (or k).  Exact mode: argmax == d_{j+1}.  Threshold mode:
// z[d_{j+1}] - z_max >= log_tau.
constexpr int kAcceptThreads = 256;
__global__ void __launch_bounds__(kAcceptThreads) accept_kernel(AcceptArgs a, RowMeta rm, const int* status) {
  pdl_wait();               // everything below reads or writes what earlier kernels of the step produced
  pdl_launch_dependents();
  const int i = blockIdx.x, tid = threadIdx.x;
  __shared__ int s_acc;
  // (three independent reads in flight together; after a failed check the two row words are unwritten and unused)
  const int failed = *status;
  const int q0 = rm.seq_q0[i], n = rm.seq_n[i];
  if (failed) {             // a failed step decides nothing: -1 makes the commit that follows leave the lengths alone
    if (tid == 0) { a.accept_len[i] = -1; a.n_emit[i] = 0; }
    return;
  }
  if (n <= 0) {
    if (tid == 0) { a.accept_len[i] = 0; a.n_emit[i] = 0; }
    return;
  }
  const int k = n - 1;
  if (tid == 0) s_acc = k;
  __syncthreads();
  int first = k;
  for (int j = tid; j < n; j += kAcceptThreads) {
    const unsigned long long best = a.row_best[q0 + j];
    const int nxt = rm.row_next[q0 + j];
    const float zd = a.zdraft[q0 + j];
    if (j < k) {
      const bool ok = a.log_tau == 0.f ? key_col(best) == nxt : zd - key_value(best) >= a.log_tau;
      if (!ok) first = min(first, j);
    }
    if (a.row_argmax) a.row_argmax[q0 + j] = key_col(best);
    if (a.row_zmax) a.row_zmax[q0 + j] = key_value(best);
    if (a.row_zdraft) a.row_zdraft[q0 + j] = zd;
  }
  if (first < k) atomicMin(&s_acc, first);
  __syncthreads();
  const int acc = s_acc;
  int* emit = a.emit_tokens + (size_t)i * a.max_q_len;
  for (int j = tid; j < acc; j += kAcceptThreads) emit[j] = rm.row_next[q0 + j];
  if (tid == 0) {
    emit[acc] = key_col(a.row_best[q0 + acc]);
    a.accept_len[i] = acc;
    a.n_emit[i] = acc + 1;
  }
}
void launch_accept(cudaStream_t st, const AcceptArgs& a, const RowMeta& rm, const int* status, bool pdl) {
  launch_kernel(accept_kernel, dim3(a.n_seqs), dim3(kAcceptThreads), 0, st, pdl, a, rm, status);
}

// ------------------------------------------------------------------------------------------------
// Greedy traversal of a candidate tree (Eq. 9-12), one CTA per sequence, one thread per node.  At the current node s:
// u_hat = the full-vocabulary argmax at s; u* = the child of s with the best score (exact mode: the child that carries
// u_hat); move to it iff z[u*] - z[u_hat] >= log tau; stop when the test fails or s has no child; emit pi(s) + u_hat.
// Every node finds its own move first, all at once; the walk is then a chase through shared memory (a step that searched
// the children with warp reductions cost ~0.7 us: 36 us for the longest of 16 paths).
__global__ void __launch_bounds__(HSD_MAX_TREE_ROWS) tree_accept_kernel(TreeAcceptArgs a, RowMeta rm, const int* status) {
  pdl_wait();               // everything below reads or writes what earlier kernels of the step produced
  pdl_launch_dependents();
  const int i = blockIdx.x, c = threadIdx.x;
  __shared__ unsigned long long s_key[HSD_MAX_TREE_ROWS];     // best (score, then lower token) among a node's children
  __shared__ unsigned long long s_best[HSD_MAX_TREE_ROWS];    // the node's own argmax word
  __shared__ int s_child[HSD_MAX_TREE_ROWS], s_tok[HSD_MAX_TREE_ROWS], s_path[HSD_MAX_TREE_ROWS], s_acc;
  const int failed = *status;
  const int q0 = rm.seq_q0[i], n = rm.seq_n[i];
  if (failed) {             // a failed step decides nothing: the compaction and the commit that follow skip -1
    if (c == 0) { a.accept_len[i] = -1; a.n_emit[i] = 0; }
    return;
  }
  if (n <= 0) {
    if (c == 0) { a.accept_len[i] = 0; a.n_emit[i] = 0; }
    return;
  }
  constexpr int kNone = 0x7fffffff;
  const bool node = c >= 1 && c < n;
  const int par = node ? a.parent[q0 + c] : -3, tok = node ? rm.row_tok[q0 + c] : -1;
  float z = node ? a.zchild[q0 + c] : 0.f;
  const unsigned long long best = c < n ? a.row_best[q0 + c] : 0ull;
  s_best[c] = best;
  s_key[c] = 0ull;
  s_child[c] = kNone;
  s_tok[c] = tok;
  __syncthreads();
  const bool child = node && par >= 0 && par < n;
  // A child's logit and its parent's maximum are summed in different orders.  The child that carries the argmax has the LM head's
  // logit for it.  Of any other the LM head has found that it is no larger than the maximum, and smaller if its id is lower: where
  // the other sum says otherwise (equal or nearly equal logits) it is held to that, so that no sibling passes the argmax.  NaN stays.
  if (child) {
    const int hat = key_col(s_best[par]);
    const float zmax = key_value(s_best[par]), most = tok < hat ? nextafterf(zmax, -INFINITY) : zmax;
    if (tok == hat) z = zmax;
    else if (z > most) z = most;
  }
  if (a.log_tau == 0.f) {
    // the child that carries u_hat (lowest row if a caller packed the same token twice under one parent)
    if (child && tok == key_col(s_best[par])) atomicMin(&s_child[par], c);
  } else {
    // best child by (score, then lower token id), then lower row among equals
    const unsigned long long key = argmax_key(z, tok);
    if (child) atomicMax(&s_key[par], key);
    __syncthreads();
    if (child && s_key[par] == key) atomicMin(&s_child[par], c);
    __syncthreads();
    const int u = s_child[c];
    if (u != kNone && !(key_value(s_key[c]) - key_value(best) >= a.log_tau)) s_child[c] = kNone;
  }
  __syncthreads();
  if (c == 0) {
    int s = 0, acc = 0;
    while (s_child[s] != kNone && acc < n) {
      s = s_child[s];
      s_path[acc++] = s;
    }
    s_acc = acc;
  }
  __syncthreads();
  const int acc = s_acc;
  int* emit = a.emit_tokens + (size_t)i * a.max_q_len;
  int* path = a.accept_rows + (size_t)i * a.max_q_len;
  if (c < acc) {
    path[c] = s_path[c];
    emit[c] = s_tok[s_path[c]];
  }
  if (c == 0) {
    emit[acc] = key_col(s_best[acc ? s_path[acc - 1] : 0]);
    a.accept_len[i] = acc;
    a.n_emit[i] = acc + 1;
  }
  if (c < n) {
    if (a.row_argmax) a.row_argmax[q0 + c] = key_col(best);
    if (a.row_zmax) a.row_zmax[q0 + c] = key_value(best);
    if (a.row_zchild) a.row_zchild[q0 + c] = c > 0 ? z : __int_as_float(0x7fc00000);
  }
}
void launch_tree_accept(cudaStream_t st, const TreeAcceptArgs& a, const RowMeta& rm, const int* status, bool pdl) {
  launch_kernel(tree_accept_kernel, dim3(a.n_seqs), dim3(HSD_MAX_TREE_ROWS), 0, st, pdl, a, rm, status);
}

// KV maintenance after a tree step (Sec. 4.2: rollbacks and cache maintenance are part of the decode loop): the
// accepted path's rows move from their packed places L + r_d to the places L + d their rotary positions stand for.
// One CTA per (sequence, layer), one thread per 16-byte chunk of a token's K and V rows, kCompactBatch depths at a time:
// a path's rows increase strictly and none lies before its place (r_d >= d), so a store to depth d can only hit the source
// of a depth below d, which the same thread has read before; the loads of later depths never depend on it.  (Depth by
// depth with a barrier between them, the launch took 19 us for a path of 22 nodes.)
constexpr int kCompactBatch = 16;
__global__ void tree_compact_kernel(KvView kv, int n_kv_heads, int head_dim, int n_seqs, const int* seq_slots,
                                    const int* accept_len, const int* accept_rows, int max_q_len) {
  pdl_wait();               // everything below reads or writes what earlier kernels of the step produced
  pdl_launch_dependents();
  const int i = blockIdx.x, layer = blockIdx.y;
  const int slot = seq_slots ? seq_slots[i] : i;
  if (slot < 0 || slot >= kv.n_slots) return;
  const int a = accept_len[i];
  if (a < 0) return;                                     // the step failed a device-side check: nothing to keep
  const int L = kv.seq_lens[slot];
  if (L < 0 || (long long)L + max_q_len > (long long)kv.max_blocks * HSD_KV_BLOCK) return;
  const int* bt = kv.block_table + (size_t)slot * kv.max_blocks;
  const int row_chunks = head_dim / 8;                   // 16-byte chunks of one (token, kv head) row
  const int chunks = n_kv_heads * 2 * row_chunks;        // ... of one token's K and V rows in a layer
  __shared__ int s_row[HSD_MAX_TREE_ROWS];               // source row of depth d (0: stays where it is)
  __shared__ int s_blk[HSD_MAX_TREE_ROWS / HSD_KV_BLOCK + 2];   // physical blocks of cache rows L .. L + 127
  const int n = min(a, max_q_len - 1), blk0 = L / HSD_KV_BLOCK;
  for (int d = threadIdx.x; d < HSD_MAX_TREE_ROWS; d += blockDim.x) {
    const int r = d >= 1 && d <= n ? accept_rows[(size_t)i * max_q_len + d - 1] : 0;
    s_row[d] = r != d && r > 0 && r < max_q_len ? r : 0;    // a row of this call (L + r is within the table, see above)
  }
  if (threadIdx.x < HSD_MAX_TREE_ROWS / HSD_KV_BLOCK + 2)
    s_blk[threadIdx.x] = blk0 + (int)threadIdx.x < kv.max_blocks ? bt[blk0 + threadIdx.x] : -1;
  __syncthreads();
  for (int t = threadIdx.x; t < chunks; t += blockDim.x) {
    const int c16 = t % row_chunks, pool = (t / row_chunks) & 1, h = t / (2 * row_chunks);
    uint4* base = reinterpret_cast<uint4*>(pool ? kv.v_pool : kv.k_pool) + c16;
    auto place = [&](int row, size_t& at) -> bool {        // 16-byte index of this thread's chunk of cache row L + row
      const int p = L + row, b = s_blk[p / HSD_KV_BLOCK - blk0];
      at = ((((size_t)layer * kv.n_blocks + b) * n_kv_heads + h) * 64 + p % HSD_KV_BLOCK) * row_chunks;
      return b >= 0 && b < kv.n_blocks;
    };
    for (int d0 = 1; d0 <= n; d0 += kCompactBatch) {
      uint4 v[kCompactBatch];
      size_t src, dst;
#pragma unroll
      for (int k = 0; k < kCompactBatch; ++k) {
        const int r = d0 + k <= n ? s_row[d0 + k] : 0;
        if (r && place(r, src)) v[k] = base[src];
      }
#pragma unroll
      for (int k = 0; k < kCompactBatch; ++k) {
        const int r = d0 + k <= n ? s_row[d0 + k] : 0;
        if (r && place(r, src) && place(d0 + k, dst)) base[dst] = v[k];
      }
    }
  }
}
void launch_tree_compact(cudaStream_t st, const KvView& kv, int n_layers, int n_kv_heads, int head_dim, int n_seqs,
                         const int* seq_slots, const int* accept_len, const int* accept_rows, int max_q_len, bool pdl) {
  launch_kernel(tree_compact_kernel, dim3(n_seqs, n_layers), dim3(128), 0, st, pdl, kv, n_kv_heads, head_dim, n_seqs, seq_slots,
                accept_len, accept_rows, max_q_len);
}

// ------------------------------------------------------------------------------------------------
// Draft-target matching and prefix-tree packing (Sec. 3.2, Eq. 5-7), one CTA per sequence.
//  1. the window takes in the tokens the last step emitted (w = the n most recent accepted tokens);
//  2. every position of the sequence's drafts where w occurs gives a candidate: the non-empty suffix after it
//     (Eq. 5, 6), in draft order then position order, at most kDsvMaxCands of them;
//  3. warp 0 grows the prefix tree level by level (Eq. 7): at depth d every live candidate moves to the child
//     that carries its d-th token, creating it while the node budget lasts; a candidate whose node cannot be
//     created stops.  Node ids are creation order, so parents precede children and the id is the packed row.
// A round of 2. tests kDsvPer positions per thread across draft borders; in 3. a lane holds candidates `lane` and
// `lane + 32`, and a level is one match over (current node, token): the lowest candidate of a group creates its node, in
// candidate order, as if they went one after another.  (Draft after draft in rounds of 128 positions and candidate after
// candidate, 16 drafts of 320 tokens took 111 us, 2 drafts 48 us.)
// Every sequence gets exactly max_rows rows: row 0 = the pending token, then the nodes, then padding rows
// (parent -2) that no traversal can enter.
constexpr int kDsvMaxCands = 64;
constexpr int kDsvMaxWindow = 8;
constexpr int kDsvThreads = 512, kDsvPer = 4, kDsvDrafts = 64;   // drafts taken together
__global__ void __launch_bounds__(kDsvThreads) dsv_build_kernel(DsvArgs a) {
  pdl_wait();               // everything below reads or writes what earlier kernels of the step produced
  pdl_launch_dependents();
  const int s = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  __shared__ int s_w[kDsvMaxWindow];
  __shared__ int s_cstart[kDsvMaxCands], s_clen[kDsvMaxCands];
  __shared__ int s_d0[kDsvDrafts], s_pos[kDsvDrafts + 1], s_cnt[kDsvThreads / 32];   // drafts: first token, first position
  __shared__ int s_ntok[HSD_MAX_TREE_ROWS], s_npar[HSD_MAX_TREE_ROWS];
  __shared__ int s_ctok[kDsvMaxCands][HSD_MAX_TREE_ROWS + 1];   // the part of every candidate a tree of this size can hold
  __shared__ int s_ncand, s_nnodes;
  const int n = a.window_n;
  if (tid == 0) {
    // window <- last n of (window ++ emitted)
    int tmp[2 * kDsvMaxWindow];
    int m = 0;
    for (int i = 0; i < n; ++i) tmp[m++] = a.window[s * n + i];
    if (a.emit_tokens && a.n_emit) {
      const int ne = a.n_emit[s];
      for (int i = max(0, ne - n); i < ne; ++i) {
        if (m == 2 * kDsvMaxWindow) {
          for (int k = 1; k < m; ++k) tmp[k - 1] = tmp[k];
          --m;
        }
        tmp[m++] = a.emit_tokens[(size_t)s * a.emit_stride + i];
      }
    }
    for (int i = 0; i < n; ++i) {
      s_w[i] = tmp[m - n + i];
      a.window[s * n + i] = s_w[i];
    }
    s_ncand = 0;
    s_nnodes = 0;
    a.cu_q[s] = s * a.max_rows;
    if (s == 0) a.cu_q[a.n_seqs] = a.n_seqs * a.max_rows;
  }
  __syncthreads();
  bool have_w = true;
  for (int i = 0; i < n; ++i) have_w = have_w && s_w[i] >= 0;
  // ---- candidates
  if (have_w) {
    // every offset is clamped to the array sizes the host passed: a malformed table shortens or drops drafts
    // whose drafts: the sequence's own, or (lane batches) those of the owner the map names; -1 or out of range = none
    const int owner = a.seq_map ? a.seq_map[s] : s;
    const bool owned = a.seq_map ? (owner >= 0 && owner < a.n_owners) : true;
    const int d_lo = owned ? min(max(a.seq_draft_off[owner], 0), a.n_drafts) : 0;
    const int d_hi = owned ? min(max(a.seq_draft_off[owner + 1], 0), a.n_drafts) : 0;
    for (int db = d_lo; db < d_hi && s_ncand < kDsvMaxCands; db += kDsvDrafts) {
      const int nd = min(kDsvDrafts, d_hi - db);
      if (warp == 0) {
        // positions a window can begin at with a non-empty suffix behind it, draft after draft
        int before = 0;
        for (int k0 = 0; k0 < nd; k0 += 32) {
          const int k = k0 + lane;
          int d0 = 0, cnt = 0;
          if (k < nd) {
            d0 = min(max(a.draft_off[db + k], 0), a.total_draft_tokens);
            cnt = max(0, min(max(a.draft_off[db + k + 1], d0), a.total_draft_tokens) - d0 - n);
          }
          int incl = cnt;
          for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
          }
          if (k < nd) {
            s_d0[k] = d0;
            s_pos[k] = before + incl - cnt;
          }
          before += __shfl_sync(0xffffffffu, incl, 31);
        }
        if (lane == 0) s_pos[nd] = before;
      }
      __syncthreads();
      const int n_pos = s_pos[nd];
      for (int v0 = 0; v0 < n_pos && s_ncand < kDsvMaxCands; v0 += kDsvThreads * kDsvPer) {
        const int v = v0 + tid * kDsvPer;
        int lo = 0, hi = nd;                              // the draft of position v: the last that begins at or before it
        while (hi - lo > 1) {
          const int mid = (lo + hi) >> 1;
          if (s_pos[mid] <= v) lo = mid; else hi = mid;
        }
        int dk[kDsvPer], hits = 0;
#pragma unroll
        for (int e = 0; e < kDsvPer; ++e) {
          while (lo + 1 < nd && s_pos[lo + 1] <= v + e) ++lo;
          dk[e] = lo;
          bool hit = v + e < n_pos;
          const int at = s_d0[lo] + (v + e - s_pos[lo]);
          for (int i = 0; hit && i < n; ++i) hit = a.draft_tokens[at + i] == s_w[i];
          hits |= (hit ? 1 : 0) << e;
        }
        int incl = __popc(hits);
        for (int o = 1; o < 32; o <<= 1) {
          const int x = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl += x;
        }
        if (lane == 31) s_cnt[warp] = incl;
        __syncthreads();
        int slot = s_ncand + incl - __popc(hits), all = 0;
        for (int w = 0; w < kDsvThreads / 32; ++w) {
          if (w < warp) slot += s_cnt[w];
          all += s_cnt[w];
        }
#pragma unroll
        for (int e = 0; e < kDsvPer; ++e) {
          if (!((hits >> e) & 1)) continue;
          if (slot < kDsvMaxCands) {
            const int j = v + e - s_pos[dk[e]];
            s_cstart[slot] = s_d0[dk[e]] + j + n;
            s_clen[slot] = s_pos[dk[e] + 1] - s_pos[dk[e]] - j;      // tokens behind the window
          }
          ++slot;
        }
        __syncthreads();
        if (tid == 0) s_ncand = min(kDsvMaxCands, s_ncand + all);
        __syncthreads();
      }
      __syncthreads();                                    // s_pos is rewritten
    }
  }
  __syncthreads();
  for (int idx = tid; idx < s_ncand * HSD_MAX_TREE_ROWS; idx += kDsvThreads) {
    const int c = idx / HSD_MAX_TREE_ROWS, d = idx % HSD_MAX_TREE_ROWS;
    s_ctok[c][d] = d < s_clen[c] ? a.draft_tokens[s_cstart[c] + d] : -1;
  }
  __syncthreads();
  // ---- prefix tree, level by level (warp 0; node ids 1.. in creation order, id 0 = root)
  if (warp == 0) {
    const int ncand = s_ncand, budget = a.max_rows - 1;
    const unsigned below = (1u << lane) - 1u;
    int nn = 0, cur[2] = {0, 0};
    bool alive[2] = {lane < ncand, lane + 32 < ncand};
    const int len[2] = {lane < ncand ? s_clen[lane] : 0, lane + 32 < ncand ? s_clen[lane + 32] : 0};
    bool apart = false;                                   // no two candidates stand on one node: they never meet again
    for (int depth = 0; depth < HSD_MAX_TREE_ROWS; ++depth) {
      alive[0] = alive[0] && depth < len[0];
      alive[1] = alive[1] && depth < len[1];
      const unsigned on0 = __ballot_sync(0xffffffffu, alive[0]), on1 = __ballot_sync(0xffffffffu, alive[1]);
      if (!(on0 | on1)) break;
      // two candidates go to the same child iff they stand on the same node and carry the same token
      const int tok0 = alive[0] ? s_ctok[lane][depth] : 0, tok1 = alive[1] ? s_ctok[lane + 32][depth] : 0;
      if (apart) {                                        // every live candidate has a child of its own
        const int id0 = nn + 1 + __popc(on0 & below), id1 = min(budget, nn + __popc(on0)) + 1 + __popc(on1 & below);
        if (alive[0] && id0 <= budget) { s_ntok[id0] = tok0; s_npar[id0] = cur[0]; }
        if (alive[1] && id1 <= budget) { s_ntok[id1] = tok1; s_npar[id1] = cur[1]; }
        alive[0] = alive[0] && id0 <= budget;
        alive[1] = alive[1] && id1 <= budget;
        cur[0] = id0;
        cur[1] = id1;
        nn = min(budget, nn + __popc(on0) + __popc(on1));
        continue;
      }
      const unsigned long long key0 = ((unsigned long long)cur[0] << 32) | (unsigned)tok0;
      const unsigned long long key1 = ((unsigned long long)cur[1] << 32) | (unsigned)tok1;
      unsigned same = 0u;
      if (alive[0]) same = __match_any_sync(on0, key0);
      __syncwarp();
      const bool lead0 = alive[0] && (same & below) == 0u;
      const unsigned leads0 = __ballot_sync(0xffffffffu, lead0);
      const int mine0 = nn + 1 + __popc(leads0 & below);
      const int id0 = __shfl_sync(0xffffffffu, mine0, alive[0] ? __ffs(same) - 1 : lane);
      if (lead0 && mine0 <= budget) { s_ntok[mine0] = tok0; s_npar[mine0] = cur[0]; }
      nn = min(budget, nn + __popc(leads0));
      apart = leads0 == on0;
      if (alive[0]) {
        alive[0] = id0 <= budget;                         // a node that could not be created ends its candidates
        cur[0] = id0;
      }
      if (on1) {
        int id1 = 0;
        for (unsigned m = leads0; m; m &= m - 1) {        // children that candidates 0..31 have just reached
          const int src = __ffs(m) - 1;
          const unsigned long long k = __shfl_sync(0xffffffffu, key0, src);
          const int id = __shfl_sync(0xffffffffu, mine0, src);
          if (alive[1] && k == key1) id1 = id;
        }
        const bool rest = alive[1] && id1 == 0;
        const unsigned onr = __ballot_sync(0xffffffffu, rest);
        unsigned same1 = 0u;
        if (rest) same1 = __match_any_sync(onr, key1);
        __syncwarp();
        const bool lead1 = rest && (same1 & below) == 0u;
        const unsigned leads1 = __ballot_sync(0xffffffffu, lead1);
        const int mine1 = nn + 1 + __popc(leads1 & below);
        const int got = __shfl_sync(0xffffffffu, mine1, rest ? __ffs(same1) - 1 : lane);
        if (rest) id1 = got;
        if (lead1 && mine1 <= budget) { s_ntok[mine1] = tok1; s_npar[mine1] = cur[1]; }
        nn = min(budget, nn + __popc(leads1));
        apart = apart && leads1 == on1;
        if (alive[1]) {
          alive[1] = id1 <= budget;
          cur[1] = id1;
        }
      }
    }
    if (lane == 0) s_nnodes = nn;
  }
  __syncthreads();
  // ---- packed rows
  const int nn = s_nnodes, pending = s_w[n - 1];
  for (int r = tid; r < a.max_rows; r += kDsvThreads) {
    const size_t o = (size_t)s * a.max_rows + r;
    if (r == 0) { a.q_tokens[o] = pending; a.parent[o] = -1; }
    else if (r <= nn) { a.q_tokens[o] = s_ntok[r]; a.parent[o] = s_npar[r]; }
    else { a.q_tokens[o] = pending; a.parent[o] = -2; }
  }
  if (tid == 0) a.n_rows[s] = nn + 1;
}
void launch_dsv_build(cudaStream_t st, const DsvArgs& a, bool pdl) {
  launch_kernel(dsv_build_kernel, dim3(a.n_seqs), dim3(kDsvThreads), 0, st, pdl, a);
}

// ------------------------------------------------------------------------------------------------
// Lane batches (Sec. 3.1, Stage 1: many regions, each decoded to its end by repeated steps).  A lane serves one
// sequence at a time; between two steps one CTA appends what every lane's sequence emitted, counts the step, retires
// the sequences that have reached their length and hands free lanes to waiting sequences in queue order.
// counters: [0] next waiting sequence, [1] sequences not finished, [2] steps taken.
__device__ void stage_assign_lanes(const StageDev& sd, const KvView& kv) {      // one thread, lanes in order
  int head = sd.counters[0], left = sd.counters[1];
  for (int i = 0; i < sd.n_lanes; ++i) {
    const int r = sd.lane_seq[i];
    if (r >= 0 && sd.out_len[r] < sd.max_new[r]) continue;                      // still decoding
    if (r >= 0) --left;                                                         // finished in this step
    int nxt = -1;
    while (head < sd.n_seqs && nxt < 0) {
      if (sd.out_len[head] < sd.max_new[head]) nxt = head; else --left;         // (a sequence of length <= 1 is done at once)
      ++head;
    }
    sd.lane_seq[i] = nxt;
    const int slot = nxt < 0 ? sd.idle_slot : (sd.seq_slot ? sd.seq_slot[nxt] : nxt);
    sd.lane_slot[i] = slot;
    for (int k = 0; k < sd.window_n; ++k) sd.window[i * sd.window_n + k] = -1;
    sd.window[i * sd.window_n + sd.window_n - 1] = nxt < 0 ? 0 : sd.first_token[nxt];
  }
  sd.counters[0] = head;
  sd.counters[1] = left;
  if (sd.idle_slot >= 0 && sd.idle_slot < kv.n_slots) kv.seq_lens[sd.idle_slot] = 0;   // idle lanes restart from an empty cache
}

__global__ void stage_begin_kernel(StageDev sd, KvView kv) {
  pdl_wait();               // everything below reads or writes what earlier kernels of the step produced
  pdl_launch_dependents();
  for (int r = threadIdx.x; r < sd.n_seqs; r += blockDim.x) {
    sd.out_tokens[(size_t)r * sd.out_stride] = sd.first_token[r];
    sd.out_len[r] = 1;
    sd.seq_steps[r] = 0;
    sd.seq_accepted[r] = 0;
  }
  for (int i = threadIdx.x; i < sd.n_lanes; i += blockDim.x) sd.lane_seq[i] = -1;
  if (threadIdx.x == 0) {
    sd.counters[0] = 0;
    sd.counters[1] = sd.n_seqs;
    sd.counters[2] = 0;
  }
  __syncthreads();
  if (threadIdx.x == 0) stage_assign_lanes(sd, kv);
}
void launch_stage_begin(cudaStream_t st, const StageDev& sd, const KvView& kv, bool pdl) {
  launch_kernel(stage_begin_kernel, dim3(1), dim3(128), 0, st, pdl, sd, kv);
}

__global__ void stage_advance_kernel(StageDev sd, KvView kv, const int* accept_len, const int* emit_tokens,
                                     const int* n_emit, int emit_stride) {
  pdl_wait();               // everything below reads or writes what earlier kernels of the step produced
  pdl_launch_dependents();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n_warps = blockDim.x >> 5;
  for (int i = warp; i < sd.n_lanes; i += n_warps) {       // one warp per lane
    const int r = sd.lane_seq[i];
    if (r < 0 || r >= sd.n_seqs) continue;
    const int a = accept_len[i];
    if (a < 0) continue;                                   // the step failed a device-side check: nothing was decided
    const int have = sd.out_len[r];
    const int room = max(0, min(sd.max_new[r], sd.out_stride) - have);
    const int take = min(max(n_emit[i], 0), room);
    for (int k = lane; k < take; k += 32) sd.out_tokens[(size_t)r * sd.out_stride + have + k] = emit_tokens[(size_t)i * emit_stride + k];
    __syncwarp();
    if (lane == 0) {
      sd.out_len[r] = have + take;
      sd.seq_steps[r] += 1;
      sd.seq_accepted[r] += min(a, room);
      // the window keeps the most recent accepted tokens, the pending one last
      const int n = sd.window_n;
      for (int k = 0; k < n; ++k) {
        const int back = n - 1 - k;                        // token `back` places before the newest
        const int idx = have + take - 1 - back;
        sd.window[i * n + k] = idx >= 0 ? sd.out_tokens[(size_t)r * sd.out_stride + idx] : -1;
      }
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    sd.counters[2] += 1;
    stage_assign_lanes(sd, kv);
  }
}
void launch_stage_advance(cudaStream_t st, const StageDev& sd, const KvView& kv, const int* accept_len,
                          const int* emit_tokens, const int* n_emit, int emit_stride, bool pdl) {
  launch_kernel(stage_advance_kernel, dim3(1), dim3(256), 0, st, pdl, sd, kv, accept_len, emit_tokens, n_emit, emit_stride);
}

// The page draft of Stage 2 (Eq. 3): the outputs of all sequences, concatenated, with their offsets.
__global__ void stage_aggregate_kernel(StageDev sd, int* draft_tokens, int capacity, int* draft_off) {
  pdl_wait();               // everything below reads or writes what earlier kernels of the step produced
  pdl_launch_dependents();
  __shared__ int s_off;
  if (threadIdx.x == 0) {
    int off = 0;
    for (int r = 0; r < sd.n_seqs; ++r) {                  // serial scan: a page has tens of regions
      draft_off[r] = off;
      off = min(capacity, off + max(0, min(sd.out_len[r], sd.out_stride)));
    }
    draft_off[sd.n_seqs] = off;
    s_off = off;
  }
  __syncthreads();
  for (int r = 0; r < sd.n_seqs; ++r) {
    const int lo = draft_off[r], n = draft_off[r + 1] - lo;
    for (int k = threadIdx.x; k < n; k += blockDim.x) draft_tokens[lo + k] = sd.out_tokens[(size_t)r * sd.out_stride + k];
  }
}
void launch_stage_aggregate(cudaStream_t st, const StageDev& sd, int* draft_tokens, int capacity, int* draft_off, bool pdl) {
  launch_kernel(stage_aggregate_kernel, dim3(1), dim3(256), 0, st, pdl, sd, draft_tokens, capacity, draft_off);
}

// Prefill epilogue: first pending token per sequence, and seq_lens += rows.
__global__ void first_token_kernel(const unsigned long long* row_best, int n_seqs, int* first_token, RowMeta rm,
                                   KvView kv, const int* status) {
  pdl_wait();               // everything below reads or writes what earlier kernels of the step produced
  pdl_launch_dependents();
  if (*status) return;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_seqs) return;
  first_token[i] = key_col(row_best[i]);
  kv.seq_lens[rm.seq_slot[i]] = rm.seq_len[i] + rm.seq_n[i];
}
void launch_first_token(cudaStream_t st, const unsigned long long* row_best, int n_seqs, int* first_token,
                        const RowMeta& rm, const KvView& kv, const int* status, bool pdl) {
  launch_kernel(first_token_kernel, dim3((n_seqs + 127) / 128), dim3(128), 0, st, pdl, row_best, n_seqs, first_token, rm,
                kv, status);
}

// ------------------------------------------------------------------------------------------------
// KV commit / rollback: the pending row and the accepted rows stay, the rest is dead and gets overwritten.
__global__ void commit_kernel(KvView kv, int n_seqs, const int* seq_slots, const int* accept_len, int* blocks_in_use) {
  pdl_wait();               // everything below reads or writes what earlier kernels of the step produced
  pdl_launch_dependents();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_seqs) return;
  const int slot = seq_slots ? seq_slots[i] : i;
  if (slot < 0 || slot >= kv.n_slots) return;
  const int a = accept_len[i];
  int L = kv.seq_lens[slot];
  if (a >= 0) L = min(L + a + 1, kv.max_blocks * HSD_KV_BLOCK);
  kv.seq_lens[slot] = L;
  if (blocks_in_use) blocks_in_use[i] = (L + HSD_KV_BLOCK - 1) / HSD_KV_BLOCK;
}
void launch_commit(cudaStream_t st, const KvView& kv, int n_seqs, const int* seq_slots, const int* accept_len,
                   int* blocks_in_use, bool pdl) {
  launch_kernel(commit_kernel, dim3((n_seqs + 127) / 128), dim3(128), 0, st, pdl, kv, n_seqs, seq_slots, accept_len,
                blocks_in_use);
}

// ------------------------------------------------------------------------------------------------
// Words between the host call's pinned staging and the workspace, 16 bytes a thread.  A kernel and not a copy command: the
// transfers are a few KB, and what the step waited for was the hand-over between kernels and the copy engine (two input
// copies and four result copies).  A kernel in the chain of programmatic launches takes one PCIe round trip.  Host call, copy
// commands / this: one small layer 99 / 80 us, 8 regions of 9 rows 0.955 / 0.933 ms, 12 regions of ~50 rows 1.300 / 1.270.
// Both areas start on 16 bytes and are padded to them.
__global__ void copy_words_kernel(int4* dst, const int4* src, long long n4) {
  pdl_wait();
  pdl_launch_dependents();
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += (long long)gridDim.x * blockDim.x) dst[i] = src[i];
}
void launch_copy_words(cudaStream_t st, int* dst, const int* src, size_t n, bool pdl) {
  const long long n4 = ((long long)n + 3) / 4;
  const long long ctas = (n4 + 255) / 256;
  launch_kernel(copy_words_kernel, dim3((unsigned)(ctas < 128 ? ctas : 128)), dim3(256), 0, st, pdl,
                reinterpret_cast<int4*>(dst), reinterpret_cast<const int4*>(src), n4);
}

}  // namespace hsd
