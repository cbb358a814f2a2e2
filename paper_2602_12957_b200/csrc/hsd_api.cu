// C ABI of the HSD verify-step library: context, workspace carving, the per-step kernel sequence.
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <new>
#include <vector>

#include "hsd_kernels.h"

using namespace hsd;

struct ProfEvent {
  int kc;
  cudaEvent_t a, b;   // recorded right before and right after the launch: every interval owns both its ends
};

// Everything a call of hsd_verify_regions_host bakes into its launches, by value: two calls with equal keys enqueue
// identical work (only the contents of the staged inputs differ), so the second one can replay the first one's graph.
struct HostCallKey {
  hsd_kv kv;
  const int* seq_slots;
  void* workspace;
  size_t ws_bytes;
  void* stream;
  int n_seqs, total_q, max_q, commit;
  float log_tau;
  int pad;
};

// The tiles of one projection for calls of up to 8,192 rows, by row class; larger calls, which take milliseconds, choose theirs.
struct TilePlan {
  static constexpr int kRows = 8192;
  TileChoice of[3 + kRows / 128];
};

struct hsd_ctx {
  hsd_model_config cfg;
  ModelDims md;
  const bf16 *embed, *lm_head, *final_norm;
  std::vector<const bf16*> attn_norm, w_qkv, w_o, ffn_norm, w_gate_up, w_down;
  std::vector<const bf16*> q_norm, k_norm;    // per layer, nullptr when the model has no per-head q/k norm
  std::vector<WeightMaps> tm_qkv, tm_o, tm_gate_up, tm_down;
  WeightMaps tm_lm_head;
  TilePlan tiles_qkv, tiles_o, tiles_gate_up, tiles_down, tiles_lm_head;
  int max_splits;     // K slices the residual-add projections may use (1 with HSD_FLAG_DETERMINISTIC)
  bool pdl;           // kernels are launched with programmatic stream serialization
  int force_bn, force_splits;   // hsd_debug_set_gemm_tile
  int pair;                     // GEMMs may run as CTA pairs
  int attn_target_items, attn_min_chunk;   // attention plan: units (share x kv head) aimed at per launch, shortest slice in KV blocks
  bool attn_fine;                          // hsd_debug_set_attn_plan has named the shortest slice
  int tap_layer, tap_which;                // hsd_debug_tap: armed for the next forward (tap_layer < 0: none)
  void* tap_dst;
  size_t tap_bytes;
  int n_sms;
  int device;
  bool simt;
  bool attn_simt;     // attention through the plain kernel (debug)
  int last_cuda_error;
  long long launches;
  long long tile_choices;       // hsd_debug_host_work: tiles chosen, weight maps encoded, GEMM kernels of its modes
  int n_weight_maps, n_gemm_kernels;
  bool profiling;
  // hsd_verify_regions_host: pinned staging and the cached graph of the last repeated call shape
  bool host_graph_ok;
  int* pin;
  size_t pin_ints;
  HostCallKey hg_key, hg_seen;
  bool hg_seen_valid;
  cudaGraphExec_t hg_exec;
  long long hg_launches;
  std::vector<ProfEvent> prof_events;
  std::vector<cudaEvent_t> event_pool;
  double prof_ms[KC_COUNT];
  long long prof_n[KC_COUNT];
};

namespace {

constexpr int kStatusWords = 16;

struct Ws {
  int* status;        // kStatusWords ints; [5] = attention shares per kv head
  AttnPlan plan;
  RowMeta rm;
  int* sel_rows;
  int2* verdict;      // what every set-up CTA found
  // device staging of hsd_verify_regions_host: [cu_q | q_tokens], and behind the status words [accept_len | n_emit |
  // emit_tokens], so that the inputs and the results are one transfer each
  int *h_in, *h_out;
  size_t h_out_ints;
  float* x;
  bf16* h;
  bf16* q;
  bf16* attn;
  bf16* act;
  float* qkv_f32;     // SIMT debug path only
  unsigned long long* row_best;
  float* zdraft;
  float* split_ws;    // attention split-KV partials: from h on, see split_quarters
  size_t bytes;
};

inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// Shortest slice of a q-tile's KV range in 64-key blocks: see make_attn_plan.  Heads of 128: a slice's result is twice the
// size, so ranges of 9 and 10 blocks stay whole too.  1 / 4 / 8 regions of 9 blocks, 8 layers, graph replays: 477 / 499 / 578 us at
// 8, 486 / 511 / 602 at 6; of 7 and 12 blocks alike; of 16 blocks 507 / 533 / 634 at 8, 504 / 529 / 634 at 6.
inline int attn_min_chunk(const ModelDims& md) { return md.D == 128 ? 8 : 6; }

// CTAs of an attention launch: as many as are resident at once
inline int attn_grid(const hsd_ctx* c) { return 2 * c->n_sms; }

inline int attn_max_tiles(const ModelDims& md, int T, int S) { return T / (128 / md.group) + S; }
// Shares of a kv head in an attention launch: one per CTA slot it has.
inline int attn_max_shares(const hsd_ctx* c) {
  const int n = attn_grid(c) / c->md.Hkv;
  return n < 1 ? 1 : (n > kAttnMaxShares ? kAttnMaxShares : n);
}
// Partial results of sliced q-tiles.  A slot holds what one slice of a q-tile leaves for every kv head: per 32-row quarter an
// fp32 accumulator row plus (reference, sum) for each row, of as many quarters as a q-tile of a call of T rows can have.
// Two slots per share are all a plan can use, 20 MB with 16 / 8 heads of 64; a small call gets what eight whole
// slices of each of its q-tiles take (one row 2.2 MB, 64 rows 4.3 MB) and its plan makes do with it.  The slots begin in the
// buffers of the normed rows and of the SwiGLU activation: the projections around the attention leave both unused while it runs.
// (Only single sequences of ~50 to 200 rows over more than ~9 k tokens would be cut finer with all the room: 63 / 100 / 160
// rows over 16,000 in 20 MB 1.28 / 1.38 / 1.50 ms, as it is 1.34 / 1.48 / 1.55.)
inline int attn_quarters(const ModelDims& md, int T) {
  const int tokens = 128 / md.group;
  return ((T < tokens ? T : tokens) * md.group + 31) / 32;
}
inline size_t quarter_bytes(const ModelDims& md) { return (size_t)md.Hkv * (md.D + 2) * 32 * sizeof(float); }   // of every kv head
inline int split_quarters(const hsd_ctx* c, int T, int S, size_t unused_bytes) {      // all slots together
  const long long most = 2ll * attn_max_shares(c) * attn_quarters(c->md, T);
  const long long small = 32ll * attn_max_tiles(c->md, T, S) + (long long)(unused_bytes / quarter_bytes(c->md));
  return (int)(most < small ? most : small);
}

Ws carve(const hsd_ctx* c, void* base, int T, int S) {
  const ModelDims& md = c->md;
  Ws w;
  size_t off = 0;
  char* p = static_cast<char*>(base);
  auto take = [&](size_t bytes) {
    void* r = p ? p + off : nullptr;
    off = align_up(off + bytes, 256);
    return r;
  };
  w.h_out_ints = 2 * (size_t)S + (size_t)S * (T < HSD_MAX_Q_LEN ? T : HSD_MAX_Q_LEN);
  w.status = static_cast<int*>(take(sizeof(int) * (kStatusWords + w.h_out_ints)));
  w.h_out = w.status ? w.status + kStatusWords : nullptr;
  w.rm.row_seq = static_cast<int*>(take(sizeof(int) * T));
  w.rm.row_pos = static_cast<int*>(take(sizeof(int) * T));
  w.rm.row_tok = static_cast<int*>(take(sizeof(int) * T));
  w.rm.row_kv = static_cast<int*>(take(sizeof(int) * T));
  w.rm.row_next = static_cast<int*>(take(sizeof(int) * T));
  w.rm.rope_cs = static_cast<float2*>(take(sizeof(float2) * (size_t)T * (md.D / 2)));
  w.rm.seq_q0 = static_cast<int*>(take(sizeof(int) * S));
  w.rm.seq_n = static_cast<int*>(take(sizeof(int) * S));
  w.rm.seq_len = static_cast<int*>(take(sizeof(int) * S));
  w.rm.seq_slot = static_cast<int*>(take(sizeof(int) * S));
  w.rm.seq_tile0 = static_cast<int*>(take(sizeof(int) * (S + 1)));
  w.rm.anc = static_cast<uint4*>(take(sizeof(uint4) * T));
  w.rm.child_src = static_cast<int*>(take(sizeof(int) * T));
  w.rm.child_tok = static_cast<int*>(take(sizeof(int) * T));
  w.sel_rows = static_cast<int*>(take(sizeof(int) * S));
  w.verdict = static_cast<int2*>(take(sizeof(int2) * (size_t)setup_ctas(T)));
  w.h_in = static_cast<int*>(take(sizeof(int) * ((size_t)S + 1 + T)));
  // a prefill's LM head runs over one row per sequence, and sequences without rows make those more than T
  const size_t lm_rows = T > S ? T : S;
  w.x = static_cast<float*>(take(sizeof(float) * (size_t)T * md.d));
  w.q = static_cast<bf16*>(take(2 * (size_t)T * md.Hq * md.D));
  w.attn = static_cast<bf16*>(take(2 * (size_t)T * md.Hq * md.D));
  w.qkv_f32 = c->simt ? static_cast<float*>(take(sizeof(float) * (size_t)T * md.qkv_out)) : nullptr;
  w.row_best = static_cast<unsigned long long*>(take(sizeof(unsigned long long) * lm_rows));
  w.zdraft = static_cast<float*>(take(sizeof(float) * T));
  const size_t h_bytes = align_up(2 * lm_rows * md.d, 256), act_bytes = align_up(2 * (size_t)T * md.ffn, 256);
  const int room = split_quarters(c, T, S, h_bytes + act_bytes);
  {
    const int mt = attn_max_tiles(md, T, S), most = attn_max_shares(c);
    w.plan.quarters = attn_quarters(md, T);
    w.plan.slots = room / w.plan.quarters;
    w.plan.max_shares = most < 16 * mt ? most : 16 * mt;
    if (w.plan.max_shares > w.plan.slots) w.plan.max_shares = w.plan.slots;
    const int shares = most < 16 * mt ? most : 16 * mt;     // (the arrays do not shrink where a q-tile gets more quarters)
    w.plan.items = static_cast<int4*>(take(sizeof(int4) * 2 * (size_t)(mt + shares)));
    w.plan.share_start = static_cast<int*>(take(sizeof(int) * (shares + 1)));
    w.plan.tile_seq = static_cast<int*>(take(sizeof(int) * mt));
    w.plan.tile_pos = static_cast<int*>(take(sizeof(int) * mt));
    w.plan.counters = static_cast<int*>(take(sizeof(int) * (size_t)room * md.Hkv));
    w.plan.first = static_cast<int4*>(take(sizeof(int4) * 3 * (size_t)attn_grid(c)));
    w.plan.n_shares = w.status ? w.status + 5 : nullptr;
    w.plan.n_kv_heads = md.Hkv;
    w.plan.grid = attn_grid(c);
  }
  w.h = static_cast<bf16*>(take(h_bytes));
  w.act = static_cast<bf16*>(take(act_bytes));
  w.split_ws = c->simt ? nullptr : reinterpret_cast<float*>(w.h);
  const size_t split = c->simt ? 0 : (size_t)room * quarter_bytes(md);
  if (split > h_bytes + act_bytes) take(split - h_bytes - act_bytes);
  w.bytes = align_up(off, 1024);
  return w;
}

struct Scope {   // brackets one launch: counts it and, when profiling, records events around it
  hsd_ctx* c;
  cudaStream_t st;
  int idx;
  // Two event records per launch.  An event between two kernels also keeps them from overlapping through
  // programmatic dependent launch, so a profiled interval is the kernel alone (as a serialising profiler sees it),
  // not its share of an overlapped step.
  Scope(hsd_ctx* c_, cudaStream_t st_, int kc) : c(c_), st(st_), idx(-1) {
    c->launches++;
    if (!c->profiling) return;
    auto take = [&](cudaEvent_t* ev) -> bool {
      if (!c->event_pool.empty()) {
        *ev = c->event_pool.back();
        c->event_pool.pop_back();
        return true;
      }
      return cudaEventCreate(ev) == cudaSuccess;
    };
    ProfEvent e;
    e.kc = kc;
    if (!take(&e.a)) return;
    if (!take(&e.b)) {
      c->event_pool.push_back(e.a);
      return;
    }
    cudaEventRecord(e.a, st);
    c->prof_events.push_back(e);
    idx = (int)c->prof_events.size() - 1;
  }
  ~Scope() {
    if (idx >= 0) cudaEventRecord(c->prof_events[idx].b, st);
  }
};

int fail_cuda(hsd_ctx* c) {
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) c->last_cuda_error = (int)e;
  return HSD_ERR_CUDA;
}

int check_cuda(hsd_ctx* c) {
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    c->last_cuda_error = (int)e;
    return HSD_ERR_CUDA;
  }
  return HSD_OK;
}

KvView kv_view(const hsd_kv* kv) {
  KvView v;
  v.k_pool = static_cast<bf16*>(kv->k_pool);
  v.v_pool = static_cast<bf16*>(kv->v_pool);
  v.n_blocks = kv->n_blocks;
  v.block_table = kv->block_table;
  v.max_blocks = kv->max_blocks_per_seq;
  v.seq_lens = kv->seq_lens;
  v.n_slots = kv->n_slots;
  return v;
}

int check_kv(const hsd_kv* kv) {
  if (!kv || !kv->k_pool || !kv->v_pool || !kv->block_table || !kv->seq_lens) return HSD_ERR_INVALID_ARG;
  if (kv->n_blocks <= 0 || kv->max_blocks_per_seq <= 0 || kv->n_slots <= 0) return HSD_ERR_INVALID_ARG;
  return HSD_OK;
}

TileChoice choose_tile(hsd_ctx* c, const GemmSm100Args& g, int force_bn, int force_splits) {
  ++c->tile_choices;
  return gemm_choose_tile(g, force_bn, force_splits);
}
TileChoice planned_tile(hsd_ctx* c, const GemmSm100Args& g, const TilePlan& plan) {
  return g.M <= TilePlan::kRows ? plan.of[gemm_row_class(g.M)] : choose_tile(c, g, 0, 0);
}
void make_tile_plan(hsd_ctx* c, TilePlan* plan, int n_out, int K, int mode) {
  GemmSm100Args g = {};
  g.n_out = n_out; g.K = K; g.mode = mode; g.n_sms = c->n_sms; g.pair = c->pair;
  g.max_splits = mode == GS_ADD_F32 ? c->max_splits : 1;
  for (int k = 0; k < 3 + TilePlan::kRows / 128; ++k) {
    g.M = gemm_class_rows(k);
    plan->of[k] = choose_tile(c, g, 0, 0);
  }
}

struct StepArgs {
  int n_seqs, total_q, max_q_len;
  bool prefill;
  const int* cu_q;
  const int* tokens;
  const int* pending;
  const int* draft;
  const void* embeds;
  const int* seq_slots;
  int slot_base;
  const int* parent;   // candidate trees: parent row within the sequence, or nullptr (chains)
};

// The decoder forward over one packed batch: rows -> residual stream x after the last layer.  `tm_h`: where the map of the
// batch's normed rows goes.
int run_layers(hsd_ctx* c, const hsd_kv* kvp, const StepArgs& a, const Ws& w, CUtensorMap& tm_h, cudaStream_t st) {
  const ModelDims& md = c->md;
  const KvView kv = kv_view(kvp);
  const int T = a.total_q;
  const int tokens_per_tile = 128 / md.group;

  // hsd_debug_tap: one armed tap is served by this forward, then disarmed
  const int tap_layer = c->tap_layer, tap_which = c->tap_which;
  c->tap_layer = -1;
  auto tap = [&](int layer, int which, const void* src, size_t bytes) -> int {
    if (layer != tap_layer || which != tap_which) return HSD_OK;
    if (bytes > c->tap_bytes) return HSD_ERR_WORKSPACE;
    return cudaMemcpyAsync(c->tap_dst, src, bytes, cudaMemcpyDeviceToDevice, st) == cudaSuccess ? HSD_OK : fail_cuda(c);
  };
  const size_t row_d = (size_t)T * md.d, row_q = (size_t)T * md.Hq * md.D;
  {
    Scope s(c, st, KC_SETUP);
    SetupArgs sa;
    sa.n_seqs = a.n_seqs;
    sa.total_q = a.total_q;
    sa.max_q_len = a.max_q_len;
    sa.vocab = md.V;
    sa.tokens_per_tile = tokens_per_tile;
    sa.cu_q = a.cu_q;
    sa.tokens = a.tokens;
    sa.pending = a.pending;
    sa.draft = a.draft;
    sa.seq_slots = a.seq_slots;
    sa.parent = a.parent;
    sa.slot_base = a.slot_base;
    sa.allow_embed_rows = a.prefill && a.embeds != nullptr;
    sa.rope_base = md.rope_base;
    sa.head_dim = md.D;
    sa.d = md.d;
    sa.table = c->embed;
    sa.embeds = static_cast<const bf16*>(a.embeds);
    sa.x = w.x;
    sa.row_best = w.row_best;
    sa.zdraft = w.zdraft;
    sa.verdict = w.verdict;
    // (a context with a fixed summation order never cuts a KV range: where the cuts fall depends on the batch)
    sa.make_plan = !c->attn_simt;
    sa.plan = w.plan;
    sa.rule.max_shares = max(1, min(w.plan.max_shares, c->attn_target_items / md.Hkv));
    sa.rule.min_chunk = c->attn_min_chunk;
    sa.rule.no_cut = c->max_splits == 1;
    sa.rule.fine = c->attn_fine;
    launch_setup_rows(st, sa, kv, w.rm, c->pdl);
  }

  CUtensorMap tm_attn, tm_act, tm_q, tm_k, tm_v, tm_x_add, tm_q_st, tm_act_st;
  if (!c->simt) {
    const uint32_t box = gemm_a_box_rows(T);
    if (make_tmap_2d(&tm_h, w.h, T, md.d, box) || make_tmap_2d(&tm_attn, w.attn, T, md.Hq * md.D, box) ||
        make_tmap_2d(&tm_act, w.act, T, md.ffn, box))
      return HSD_ERR_CUDA;
    // epilogue targets: residual stream (fp32 reduce-add), q and the SwiGLU activation (bf16 stores)
    if (make_tmap_2d_f32(&tm_x_add, w.x, T, md.d, 32) || make_tmap_2d(&tm_q_st, w.q, T, md.Hq * md.D, 32) ||
        make_tmap_2d(&tm_act_st, w.act, T, md.ffn, 32))
      return HSD_ERR_CUDA;
    // q as [T][Hq][D]: one box = (128/group) tokens x group heads x 64 dims -> a 128-row MMA operand (head_dim 128:
    // two boxes, one per half of the dims)
    if (make_tmap_3d(&tm_q, w.q, md.D, md.Hq, T, (uint64_t)md.D * 2, (uint64_t)md.Hq * md.D * 2, 64, md.group,
                     tokens_per_tile))
      return HSD_ERR_CUDA;
    // K / V pools as 2-D [rows, D]: one (layer, block, kv head) tile = 64 consecutive rows, fetched 64 dims at a time
    const uint64_t pool_rows = (uint64_t)md.n_layers * kv.n_blocks * md.Hkv * 64;
    if (make_tmap_2d(&tm_k, kv.k_pool, pool_rows, md.D, 64) || make_tmap_2d(&tm_v, kv.v_pool, pool_rows, md.D, 64))
      return HSD_ERR_CUDA;
  }

  // what the projections of every layer have in common, the tiles among it
  GemmSm100Args g_qkv = {}, g_o = {}, g_gate_up = {}, g_down = {};
  if (!c->simt) {
    auto projection = [&](GemmSm100Args& g, const CUtensorMap& tmA, const CUtensorMap& tmC, int n_out, int K, int mode, int max_splits,
                          const TilePlan& plan) {
      g.tmA = tmA;
      g.tmC = tmC;
      g.M = T; g.n_out = n_out; g.K = K; g.mode = mode;
      g.status = w.status; g.n_sms = c->n_sms; g.max_splits = max_splits; g.pdl = c->pdl; g.pair = c->pair;
      g.tile = planned_tile(c, g, plan);
    };
    projection(g_qkv, tm_h, tm_q_st, md.qkv_out, md.d, md.D == 128 ? GS_QKV_ROPE128 : GS_QKV_ROPE, 1, c->tiles_qkv);
    if (c->force_bn) g_qkv.tile = choose_tile(c, g_qkv, c->force_bn, 0);
    g_qkv.qkv.row_kv = w.rm.row_kv;
    g_qkv.qkv.kv_rows = kv.n_blocks * HSD_KV_BLOCK;
    g_qkv.qkv.rope_cs = w.rm.rope_cs;
    g_qkv.qkv.q_out = w.q;
    g_qkv.qkv.Hq = md.Hq; g_qkv.qkv.Hkv = md.Hkv; g_qkv.qkv.D = md.D;
    g_qkv.qkv.eps = md.eps;
    projection(g_o, tm_attn, tm_x_add, md.d, md.Hq * md.D, GS_ADD_F32, c->max_splits, c->tiles_o);
    projection(g_gate_up, tm_h, tm_act_st, 2 * md.ffn, md.d, GS_SWIGLU, 1, c->tiles_gate_up);
    g_gate_up.out.C = w.act; g_gate_up.out.ldc = md.ffn;
    projection(g_down, tm_act, tm_x_add, md.d, md.ffn, GS_ADD_F32, c->max_splits, c->tiles_down);
  }

  for (int l = 0; l < md.n_layers; ++l) {
    {
      Scope s(c, st, KC_RMSNORM);
      if (l == 0) launch_first_rmsnorm(st, w.x, c->attn_norm[l], w.h, T, md.d, md.eps, w.verdict, setup_ctas(T), w.status, c->n_sms, c->pdl);
      else launch_rmsnorm(st, w.x, c->attn_norm[l], w.h, T, md.d, md.eps, nullptr, T, w.status, c->n_sms, c->pdl);
    }
    if (int rc = tap(l, HSD_TAP_H_ATTN, w.h, 2 * row_d)) return rc;
    const size_t layer_elems = (size_t)kv.n_blocks * md.Hkv * 64 * md.D;
    if (c->simt) {
      {
        Scope s(c, st, KC_GEMM_QKV);
        GemmOut o = {w.qkv_f32, md.qkv_out, nullptr, nullptr, nullptr};
        launch_gemm_simt(st, w.h, c->w_qkv[l], T, md.qkv_out, md.d, GM_STORE_F32, o);
      }
      {
        Scope s(c, st, KC_ROPE_KV);
        launch_rope_kvwrite(st, w.qkv_f32, w.rm, kv, md, l, w.q, T, w.status, c->q_norm[l], c->k_norm[l]);
      }
      {
        Scope s(c, st, KC_ATTN);
        launch_attn_simt(st, w.q, w.rm, kv, md, l, w.attn, T, w.status);
      }
      {
        Scope s(c, st, KC_GEMM_O);
        GemmOut o = {w.x, md.d, nullptr, nullptr, nullptr};
        launch_gemm_simt(st, w.attn, c->w_o[l], T, md.d, md.Hq * md.D, GM_ADD_F32, o);
      }
    } else {
      {
        Scope s(c, st, KC_GEMM_QKV);
        g_qkv.tmB = &c->tm_qkv[l];
        g_qkv.qkv.k_pool_layer = kv.k_pool + (size_t)l * layer_elems;
        g_qkv.qkv.v_pool_layer = kv.v_pool + (size_t)l * layer_elems;
        g_qkv.qkv.q_norm = c->q_norm[l]; g_qkv.qkv.k_norm = c->k_norm[l];
        if (launch_gemm_sm100(st, g_qkv)) return fail_cuda(c);
      }
      {
        Scope s(c, st, KC_ATTN);
        if (c->attn_simt) {
          launch_attn_simt(st, w.q, w.rm, kv, md, l, w.attn, T, w.status);
        } else if (launch_attn_sm100(st, tm_q, tm_k, tm_v, w.plan, kv, md, l, w.attn, c->device, w.status, w.split_ws,
                                     a.parent ? w.rm.anc : nullptr, c->pdl)) {
          return fail_cuda(c);
        }
      }
      {
        Scope s(c, st, KC_GEMM_O);
        g_o.tmB = &c->tm_o[l];
        if (launch_gemm_sm100(st, g_o)) return fail_cuda(c);
      }
    }
    if (int rc = tap(l, HSD_TAP_Q, w.q, 2 * row_q)) return rc;
    if (int rc = tap(l, HSD_TAP_ATTN, w.attn, 2 * row_q)) return rc;
    if (int rc = tap(l, HSD_TAP_X_MID, w.x, 4 * row_d)) return rc;
    {
      Scope s(c, st, KC_RMSNORM);
      launch_rmsnorm(st, w.x, c->ffn_norm[l], w.h, T, md.d, md.eps, nullptr, T, w.status, c->n_sms, c->pdl);
    }
    if (int rc = tap(l, HSD_TAP_H_FFN, w.h, 2 * row_d)) return rc;
    if (c->simt) {
      {
        Scope s(c, st, KC_GEMM_GATEUP);
        GemmOut o = {w.act, md.ffn, nullptr, nullptr, nullptr};
        launch_gemm_simt(st, w.h, c->w_gate_up[l], T, 2 * md.ffn, md.d, GM_SWIGLU, o);
      }
      {
        Scope s(c, st, KC_GEMM_DOWN);
        GemmOut o = {w.x, md.d, nullptr, nullptr, nullptr};
        launch_gemm_simt(st, w.act, c->w_down[l], T, md.d, md.ffn, GM_ADD_F32, o);
      }
    } else {
      {
        Scope s(c, st, KC_GEMM_GATEUP);
        g_gate_up.tmB = &c->tm_gate_up[l];
        if (launch_gemm_sm100(st, g_gate_up)) return fail_cuda(c);
      }
      {
        Scope s(c, st, KC_GEMM_DOWN);
        g_down.tmB = &c->tm_down[l];
        if (launch_gemm_sm100(st, g_down)) return fail_cuda(c);
      }
    }
    if (int rc = tap(l, HSD_TAP_ACT, w.act, 2 * (size_t)T * md.ffn)) return rc;
    if (int rc = tap(l, HSD_TAP_X, w.x, 4 * row_d)) return rc;
  }
  return check_cuda(c);
}

// LM head + running argmax over `rows` rows of h (already selected / normalised into w.h); the set-up kernel cleared them.
// `tm_h`: run_layers' map of h, where the rows are the batch's, or nullptr.
int run_lm_head(hsd_ctx* c, const Ws& w, int rows, const CUtensorMap* tm_h, const int* row_next, cudaStream_t st) {
  const ModelDims& md = c->md;
  Scope s(c, st, KC_LMHEAD);
  GemmOut o = {nullptr, 0, w.row_best, w.zdraft, row_next};
  if (c->simt) {
    launch_gemm_simt(st, w.h, c->lm_head, rows, md.V, md.d, GM_ARGMAX, o);
  } else {
    GemmSm100Args g = {};
    if (tm_h) g.tmA = *tm_h;
    else if (make_tmap_2d(&g.tmA, w.h, rows, md.d, gemm_a_box_rows(rows))) return HSD_ERR_CUDA;
    g.tmB = &c->tm_lm_head;
    g.M = rows; g.n_out = md.V; g.K = md.d; g.mode = GS_ARGMAX;
    g.out = o;
    g.status = w.status; g.n_sms = c->n_sms; g.max_splits = 1; g.pdl = c->pdl; g.pair = c->pair;
    g.tile = planned_tile(c, g, c->tiles_lm_head);
    if (launch_gemm_sm100(st, g)) return fail_cuda(c);
  }
  return check_cuda(c);
}

int check_ws(const hsd_ctx* c, void* workspace, size_t ws_bytes, int T, int S) {
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 1023)) return HSD_ERR_WORKSPACE;
  if (hsd_workspace_bytes(c, T, S) > ws_bytes) return HSD_ERR_WORKSPACE;
  return HSD_OK;
}

int verify_common(hsd_ctx* c, const hsd_kv* kv, const StepArgs& a, float log_tau, int* accept_len, int* emit_tokens,
                  int* n_emit, int* row_argmax, float* row_zmax, float* row_zdraft, void* workspace, size_t ws_bytes,
                  cudaStream_t st) {
  int rc = check_ws(c, workspace, ws_bytes, a.total_q, a.n_seqs);
  if (rc) return rc;
  const Ws w = carve(c, workspace, a.total_q, a.n_seqs);
  CUtensorMap tm_h;
  rc = run_layers(c, kv, a, w, tm_h, st);
  if (rc) return rc;
  {
    Scope s(c, st, KC_RMSNORM);
    launch_rmsnorm(st, w.x, c->final_norm, w.h, a.total_q, c->md.d, c->md.eps, nullptr, a.total_q, w.status, c->n_sms, c->pdl);
  }
  rc = run_lm_head(c, w, a.total_q, &tm_h, w.rm.row_next, st);
  if (rc) return rc;
  {
    Scope s(c, st, KC_ACCEPT);
    AcceptArgs aa;
    aa.n_seqs = a.n_seqs;
    aa.max_q_len = a.max_q_len;
    aa.log_tau = log_tau;
    aa.row_best = w.row_best;
    aa.zdraft = w.zdraft;
    aa.accept_len = accept_len;
    aa.emit_tokens = emit_tokens;
    aa.n_emit = n_emit;
    aa.row_argmax = row_argmax;
    aa.row_zmax = row_zmax;
    aa.row_zdraft = row_zdraft;
    launch_accept(st, aa, w.rm, w.status, c->pdl);
  }
  return check_cuda(c);
}

}  // namespace

// =================================================================================================
extern "C" {

const char* hsd_status_string(int s) {
  switch (s) {
    case HSD_OK: return "ok";
    case HSD_ERR_INVALID_ARG: return "invalid argument";
    case HSD_ERR_SHAPE: return "unsupported model shape";
    case HSD_ERR_TOO_LONG: return "sequence has too many query rows";
    case HSD_ERR_WORKSPACE: return "workspace too small or misaligned";
    case HSD_ERR_KV_CAPACITY: return "KV capacity exceeded";
    case HSD_ERR_CUDA: return "CUDA error";
    case HSD_ERR_DEVICE_CHECK: return "device-side check failed";
    case HSD_ERR_NO_DEVICE: return "no usable sm_100 device";
    default: return "unknown status";
  }
}

int hsd_create(const hsd_model_config* cfg, const hsd_weights* w, hsd_ctx** out) {
  if (!cfg || !w || !out) return HSD_ERR_INVALID_ARG;
  *out = nullptr;
  if (cfg->n_layers <= 0 || cfg->d_model <= 0 || cfg->n_heads <= 0 || cfg->n_kv_heads <= 0 || cfg->d_ffn <= 0 ||
      cfg->vocab <= 0)
    return HSD_ERR_INVALID_ARG;
  if ((cfg->head_dim != 64 && cfg->head_dim != 128) || cfg->kv_block != HSD_KV_BLOCK) return HSD_ERR_SHAPE;
  // the plain cross-check kernels exist for head_dim 64 only
  if (cfg->head_dim != 64 && (cfg->flags & (HSD_FLAG_SIMT_DEBUG | HSD_FLAG_SIMT_ATTENTION))) return HSD_ERR_SHAPE;
  if (cfg->n_heads % cfg->n_kv_heads) return HSD_ERR_SHAPE;
  const int group = cfg->n_heads / cfg->n_kv_heads;
  if (128 % group) return HSD_ERR_SHAPE;
  const int dv = cfg->d_model / 128;
  if (cfg->d_model % 128 || !(dv == 1 || dv == 2 || dv == 4 || dv == 8 || dv == 16 || dv == 32)) return HSD_ERR_SHAPE;
  if (cfg->d_ffn % 64 || cfg->vocab % 64) return HSD_ERR_SHAPE;
  if (!w->embed || !w->lm_head || !w->final_norm || !w->attn_norm || !w->w_qkv || !w->w_o || !w->ffn_norm ||
      !w->w_gate_up || !w->w_down)
    return HSD_ERR_INVALID_ARG;
  for (int l = 0; l < cfg->n_layers; ++l)
    if (!w->attn_norm[l] || !w->w_qkv[l] || !w->w_o[l] || !w->ffn_norm[l] || !w->w_gate_up[l] || !w->w_down[l])
      return HSD_ERR_INVALID_ARG;
  if (cfg->qk_norm) {
    if (!w->q_norm || !w->k_norm) return HSD_ERR_INVALID_ARG;
    for (int l = 0; l < cfg->n_layers; ++l)
      if (!w->q_norm[l] || !w->k_norm[l]) return HSD_ERR_INVALID_ARG;
  }

  int dev = 0;
  int major = 0, n_sms = 0;      // (the two attributes alone: cudaGetDeviceProperties took 2.3 of a context's 2.5 ms)
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&n_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return HSD_ERR_NO_DEVICE;
  if (major != 10) return HSD_ERR_NO_DEVICE;

  hsd_ctx* c = new (std::nothrow) hsd_ctx();
  if (!c) return HSD_ERR_INVALID_ARG;
  c->cfg = *cfg;
  ModelDims& md = c->md;
  md.n_layers = cfg->n_layers; md.d = cfg->d_model; md.Hq = cfg->n_heads; md.Hkv = cfg->n_kv_heads; md.D = cfg->head_dim;
  md.ffn = cfg->d_ffn; md.V = cfg->vocab; md.qkv_out = (md.Hq + 2 * md.Hkv) * md.D; md.group = group;
  md.rope_base = cfg->rope_base; md.eps = cfg->rms_eps;
  c->embed = static_cast<const bf16*>(w->embed);
  c->lm_head = static_cast<const bf16*>(w->lm_head);
  c->final_norm = static_cast<const bf16*>(w->final_norm);
  for (int l = 0; l < md.n_layers; ++l) {
    c->attn_norm.push_back(static_cast<const bf16*>(w->attn_norm[l]));
    c->w_qkv.push_back(static_cast<const bf16*>(w->w_qkv[l]));
    c->w_o.push_back(static_cast<const bf16*>(w->w_o[l]));
    c->ffn_norm.push_back(static_cast<const bf16*>(w->ffn_norm[l]));
    c->w_gate_up.push_back(static_cast<const bf16*>(w->w_gate_up[l]));
    c->w_down.push_back(static_cast<const bf16*>(w->w_down[l]));
    c->q_norm.push_back(cfg->qk_norm ? static_cast<const bf16*>(w->q_norm[l]) : nullptr);
    c->k_norm.push_back(cfg->qk_norm ? static_cast<const bf16*>(w->k_norm[l]) : nullptr);
  }
  c->n_sms = n_sms;
  c->device = dev;
  c->simt = (cfg->flags & HSD_FLAG_SIMT_DEBUG) != 0;
  c->attn_simt = c->simt || (cfg->flags & HSD_FLAG_SIMT_ATTENTION) != 0;
  c->max_splits = (cfg->flags & HSD_FLAG_DETERMINISTIC) ? 1 : 8;
  c->pdl = (cfg->flags & HSD_FLAG_NO_PDL) == 0;
  c->force_bn = c->force_splits = 0;
  c->pair = (cfg->flags & HSD_FLAG_NO_PAIR) == 0;
  c->host_graph_ok = (cfg->flags & HSD_FLAG_NO_HOST_GRAPH) == 0;
  c->pin = nullptr;
  c->pin_ints = 0;
  c->hg_seen_valid = false;
  c->hg_exec = nullptr;
  c->hg_launches = 0;
  c->attn_target_items = attn_grid(c);
  c->attn_min_chunk = attn_min_chunk(c->md);
  c->attn_fine = false;
  c->tap_layer = -1; c->tap_which = 0; c->tap_dst = nullptr; c->tap_bytes = 0;
  c->last_cuda_error = 0;
  c->launches = 0;
  c->tile_choices = 0;
  c->n_weight_maps = c->n_gemm_kernels = 0;
  c->profiling = false;
  memset(c->prof_ms, 0, sizeof(c->prof_ms));
  memset(c->prof_n, 0, sizeof(c->prof_n));
  if (!c->simt) {
    const int qkv_mode = md.D == 128 ? GS_QKV_ROPE128 : GS_QKV_ROPE;
    int bad = tma_init();
    for (int mode : {qkv_mode, (int)GS_ADD_F32, (int)GS_SWIGLU, (int)GS_ARGMAX}) bad = bad || gemm_sm100_prepare(mode, &c->n_gemm_kernels);
    if (bad) { delete c; return HSD_ERR_CUDA; }
    c->tm_qkv.resize(md.n_layers); c->tm_o.resize(md.n_layers);
    c->tm_gate_up.resize(md.n_layers); c->tm_down.resize(md.n_layers);
    int* n = &c->n_weight_maps;
    for (int l = 0; l < md.n_layers; ++l) {
      bad |= make_weight_tmaps(&c->tm_qkv[l], c->w_qkv[l], md.qkv_out, md.d, qkv_mode, n);
      bad |= make_weight_tmaps(&c->tm_o[l], c->w_o[l], md.d, md.Hq * md.D, GS_ADD_F32, n);
      bad |= make_weight_tmaps(&c->tm_gate_up[l], c->w_gate_up[l], 2 * md.ffn, md.d, GS_SWIGLU, n);
      bad |= make_weight_tmaps(&c->tm_down[l], c->w_down[l], md.d, md.ffn, GS_ADD_F32, n);
    }
    bad |= make_weight_tmaps(&c->tm_lm_head, c->lm_head, md.V, md.d, GS_ARGMAX, n);
    if (bad) { delete c; return HSD_ERR_CUDA; }
    make_tile_plan(c, &c->tiles_qkv, md.qkv_out, md.d, qkv_mode);
    make_tile_plan(c, &c->tiles_o, md.d, md.Hq * md.D, GS_ADD_F32);
    make_tile_plan(c, &c->tiles_gate_up, 2 * md.ffn, md.d, GS_SWIGLU);
    make_tile_plan(c, &c->tiles_down, md.d, md.ffn, GS_ADD_F32);
    make_tile_plan(c, &c->tiles_lm_head, md.V, md.d, GS_ARGMAX);
  }
  *out = c;
  return HSD_OK;
}

int hsd_destroy(hsd_ctx* c) {
  if (!c) return HSD_ERR_INVALID_ARG;
  for (auto& e : c->prof_events) { cudaEventDestroy(e.a); cudaEventDestroy(e.b); }
  for (auto& e : c->event_pool) cudaEventDestroy(e);
  if (c->hg_exec) cudaGraphExecDestroy(c->hg_exec);
  if (c->pin) cudaFreeHost(c->pin);
  delete c;
  return HSD_OK;
}

size_t hsd_workspace_bytes(const hsd_ctx* c, int max_total_q, int max_seqs) {
  if (!c || max_total_q <= 0 || max_seqs <= 0) return 0;
  return carve(c, nullptr, max_total_q, max_seqs).bytes;
}

int hsd_prefill(hsd_ctx* c, const hsd_kv* kv, int n_seqs, const int* cu_len, const void* embeds, const int* token_ids,
                const int* seq_slots, int total_rows, int max_len, int* first_token, void* workspace, size_t ws_bytes,
                void* cuda_stream) {
  if (!c || !cu_len || !token_ids || !first_token) return HSD_ERR_INVALID_ARG;
  if (n_seqs <= 0 || total_rows <= 0 || max_len <= 0 || max_len > total_rows) return HSD_ERR_INVALID_ARG;
  if (max_len > 32768) return HSD_ERR_TOO_LONG;
  int rc = check_kv(kv);
  if (rc) return rc;
  if ((long long)max_len > (long long)kv->max_blocks_per_seq * HSD_KV_BLOCK) return HSD_ERR_KV_CAPACITY;
  rc = check_ws(c, workspace, ws_bytes, total_rows, n_seqs);
  if (rc) return rc;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  const Ws w = carve(c, workspace, total_rows, n_seqs);
  StepArgs a = {};
  a.n_seqs = n_seqs; a.total_q = total_rows; a.max_q_len = max_len; a.prefill = true;
  a.cu_q = cu_len; a.tokens = token_ids; a.embeds = embeds; a.seq_slots = seq_slots; a.slot_base = 0;
  CUtensorMap tm_h;
  rc = run_layers(c, kv, a, w, tm_h, st);
  if (rc) return rc;
  {
    Scope s(c, st, KC_RMSNORM);
    launch_select_last_rows(st, w.rm, n_seqs, w.sel_rows, w.status, c->pdl);
  }
  {
    Scope s(c, st, KC_RMSNORM);
    launch_rmsnorm(st, w.x, c->final_norm, w.h, n_seqs, c->md.d, c->md.eps, w.sel_rows, total_rows, w.status, c->n_sms, c->pdl);
  }
  rc = run_lm_head(c, w, n_seqs, nullptr, nullptr, st);
  if (rc) return rc;
  {
    Scope s(c, st, KC_ACCEPT);
    launch_first_token(st, w.row_best, n_seqs, first_token, w.rm, kv_view(kv), w.status, c->pdl);
  }
  return check_cuda(c);
}

int hsd_verify_regions(hsd_ctx* c, const hsd_kv* kv, int n_seqs, const int* cu_q, const int* q_tokens,
                       const int* seq_slots, int max_q_len, int total_q, float log_tau, int* accept_len,
                       int* emit_tokens, int* n_emit, int* row_argmax, float* row_zmax, float* row_zdraft,
                       void* workspace, size_t ws_bytes, void* cuda_stream) {
  if (!c || !cu_q || !q_tokens || !accept_len || !emit_tokens || !n_emit) return HSD_ERR_INVALID_ARG;
  if (n_seqs <= 0 || total_q <= 0 || max_q_len <= 0 || max_q_len > total_q) return HSD_ERR_INVALID_ARG;
  if (!(log_tau <= 0.f)) return HSD_ERR_INVALID_ARG;
  if (max_q_len > HSD_MAX_Q_LEN) return HSD_ERR_TOO_LONG;
  int rc = check_kv(kv);
  if (rc) return rc;
  if ((long long)max_q_len > (long long)kv->max_blocks_per_seq * HSD_KV_BLOCK) return HSD_ERR_KV_CAPACITY;
  StepArgs a = {};
  a.n_seqs = n_seqs; a.total_q = total_q; a.max_q_len = max_q_len; a.prefill = false;
  a.cu_q = cu_q; a.tokens = q_tokens; a.seq_slots = seq_slots; a.slot_base = 0;
  return verify_common(c, kv, a, log_tau, accept_len, emit_tokens, n_emit, row_argmax, row_zmax, row_zdraft, workspace,
                       ws_bytes, static_cast<cudaStream_t>(cuda_stream));
}

int hsd_verify_tree(hsd_ctx* c, const hsd_kv* kv, int n_seqs, const int* cu_q, const int* q_tokens, const int* parent,
                    const int* seq_slots, int max_q_len, int total_q, float log_tau, int* accept_len, int* emit_tokens,
                    int* n_emit, int* accept_rows, int* row_argmax, float* row_zmax, float* row_zchild, void* workspace,
                    size_t ws_bytes, void* cuda_stream) {
  if (!c || !cu_q || !q_tokens || !parent || !accept_len || !emit_tokens || !n_emit || !accept_rows)
    return HSD_ERR_INVALID_ARG;
  if (n_seqs <= 0 || total_q <= 0 || max_q_len <= 0 || max_q_len > total_q) return HSD_ERR_INVALID_ARG;
  if (!(log_tau <= 0.f)) return HSD_ERR_INVALID_ARG;
  if (max_q_len > HSD_MAX_TREE_ROWS) return HSD_ERR_TOO_LONG;
  if (c->simt || c->attn_simt) return HSD_ERR_INVALID_ARG;   // the plain debug kernels know chains only
  int rc = check_kv(kv);
  if (rc) return rc;
  if ((long long)max_q_len > (long long)kv->max_blocks_per_seq * HSD_KV_BLOCK) return HSD_ERR_KV_CAPACITY;
  // (sized for 2 x total_q rows, as its contract has it)
  rc = check_ws(c, workspace, ws_bytes, 2 * total_q, n_seqs);
  if (rc) return rc;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  const Ws w = carve(c, workspace, 2 * total_q, n_seqs);
  StepArgs a = {};
  a.n_seqs = n_seqs; a.total_q = total_q; a.max_q_len = max_q_len; a.prefill = false;
  a.cu_q = cu_q; a.tokens = q_tokens; a.seq_slots = seq_slots; a.slot_base = 0; a.parent = parent;
  CUtensorMap tm_h;
  rc = run_layers(c, kv, a, w, tm_h, st);
  if (rc) return rc;
  {
    Scope s(c, st, KC_RMSNORM);
    launch_tree_final_norm(st, w.x, c->final_norm, w.h, total_q, c->md.d, c->md.eps, w.rm, c->lm_head, c->md.V, w.zdraft, w.status,
                           c->pdl);
  }
  rc = run_lm_head(c, w, total_q, &tm_h, nullptr, st);
  if (rc) return rc;
  {
    Scope s(c, st, KC_ACCEPT);
    TreeAcceptArgs ta;
    ta.n_seqs = n_seqs; ta.max_q_len = max_q_len; ta.log_tau = log_tau;
    ta.parent = parent;
    ta.row_best = w.row_best;
    ta.zchild = w.zdraft;
    ta.accept_len = accept_len; ta.emit_tokens = emit_tokens; ta.n_emit = n_emit; ta.accept_rows = accept_rows;
    ta.row_argmax = row_argmax; ta.row_zmax = row_zmax; ta.row_zchild = row_zchild;
    launch_tree_accept(st, ta, w.rm, w.status, c->pdl);
  }
  return check_cuda(c);
}

int hsd_dsv_build(hsd_ctx* c, int n_seqs, int window_n, int* window, const int* emit_tokens, const int* n_emit,
                  int emit_stride, const int* draft_tokens, int total_draft_tokens, const int* draft_off, int n_drafts,
                  const int* seq_draft_off, int max_rows, int* q_tokens, int* parent, int* cu_q, int* n_rows,
                  const int* seq_map, int n_owners, void* cuda_stream) {
  if (!c || !window || !draft_tokens || !draft_off || !seq_draft_off || !q_tokens || !parent || !cu_q || !n_rows)
    return HSD_ERR_INVALID_ARG;
  if (n_seqs <= 0 || window_n <= 0 || window_n > HSD_MAX_WINDOW || max_rows <= 0) return HSD_ERR_INVALID_ARG;
  if (total_draft_tokens < 0 || n_drafts < 0) return HSD_ERR_INVALID_ARG;
  if ((emit_tokens == nullptr) != (n_emit == nullptr) || (emit_tokens && emit_stride <= 0)) return HSD_ERR_INVALID_ARG;
  if (max_rows > HSD_MAX_TREE_ROWS) return HSD_ERR_TOO_LONG;
  if (seq_map && n_owners < 0) return HSD_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  Scope s(c, st, KC_SETUP);
  DsvArgs a;
  a.seq_map = seq_map; a.n_owners = seq_map ? n_owners : n_seqs;
  a.n_seqs = n_seqs; a.window_n = window_n; a.max_rows = max_rows; a.emit_stride = emit_stride;
  a.window = window; a.emit_tokens = emit_tokens; a.n_emit = n_emit;
  a.draft_tokens = draft_tokens; a.draft_off = draft_off; a.seq_draft_off = seq_draft_off;
  a.total_draft_tokens = total_draft_tokens; a.n_drafts = n_drafts;
  a.q_tokens = q_tokens; a.parent = parent; a.cu_q = cu_q; a.n_rows = n_rows;
  launch_dsv_build(st, a, c->pdl);
  return check_cuda(c);
}

namespace {
int stage_dev(const hsd_stage* s, StageDev* d) {
  if (!s || !s->lane_seq || !s->lane_slot || !s->window || !s->first_token || !s->max_new || !s->out_tokens ||
      !s->out_len || !s->seq_steps || !s->seq_accepted || !s->counters)
    return HSD_ERR_INVALID_ARG;
  if (s->n_lanes < 1 || s->n_seqs < 1 || s->out_stride < 1 || s->window_n < 1 || s->window_n > HSD_MAX_WINDOW)
    return HSD_ERR_INVALID_ARG;
  d->n_lanes = s->n_lanes; d->n_seqs = s->n_seqs; d->window_n = s->window_n; d->out_stride = s->out_stride;
  d->idle_slot = s->idle_slot;
  d->lane_seq = s->lane_seq; d->lane_slot = s->lane_slot; d->window = s->window;
  d->first_token = s->first_token; d->seq_slot = s->seq_slot; d->max_new = s->max_new;
  d->out_tokens = s->out_tokens; d->out_len = s->out_len; d->seq_steps = s->seq_steps;
  d->seq_accepted = s->seq_accepted; d->counters = s->counters;
  return HSD_OK;
}
}  // namespace

int hsd_stage_begin(hsd_ctx* c, const hsd_stage* stage, const hsd_kv* kv, void* cuda_stream) {
  if (!c) return HSD_ERR_INVALID_ARG;
  StageDev d;
  int rc = stage_dev(stage, &d);
  if (rc) return rc;
  rc = check_kv(kv);
  if (rc) return rc;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  Scope s(c, st, KC_SETUP);
  launch_stage_begin(st, d, kv_view(kv), c->pdl);
  return check_cuda(c);
}

int hsd_stage_advance(hsd_ctx* c, const hsd_stage* stage, const hsd_kv* kv, const int* accept_len, const int* emit_tokens,
                      const int* n_emit, int emit_stride, void* cuda_stream) {
  if (!c || !accept_len || !emit_tokens || !n_emit || emit_stride < 1) return HSD_ERR_INVALID_ARG;
  StageDev d;
  int rc = stage_dev(stage, &d);
  if (rc) return rc;
  rc = check_kv(kv);
  if (rc) return rc;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  Scope s(c, st, KC_COMMIT);
  launch_stage_advance(st, d, kv_view(kv), accept_len, emit_tokens, n_emit, emit_stride, c->pdl);
  return check_cuda(c);
}

int hsd_stage_aggregate(hsd_ctx* c, const hsd_stage* stage, int* draft_tokens, int capacity, int* draft_off,
                        void* cuda_stream) {
  if (!c || !draft_tokens || !draft_off || capacity < 1) return HSD_ERR_INVALID_ARG;
  StageDev d;
  int rc = stage_dev(stage, &d);
  if (rc) return rc;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  Scope s(c, st, KC_SETUP);
  launch_stage_aggregate(st, d, draft_tokens, capacity, draft_off, c->pdl);
  return check_cuda(c);
}

int hsd_kv_commit_tree(hsd_ctx* c, const hsd_kv* kv, int n_seqs, const int* seq_slots, const int* accept_len,
                       const int* accept_rows, int max_q_len, int* blocks_in_use, void* cuda_stream) {
  if (!c || !accept_len || !accept_rows || n_seqs <= 0 || max_q_len <= 0 || max_q_len > HSD_MAX_TREE_ROWS)
    return HSD_ERR_INVALID_ARG;
  int rc = check_kv(kv);
  if (rc) return rc;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  {
    Scope s(c, st, KC_COMMIT);
    launch_tree_compact(st, kv_view(kv), c->md.n_layers, c->md.Hkv, c->md.D, n_seqs, seq_slots, accept_len, accept_rows, max_q_len,
                        c->pdl);
  }
  {
    Scope s(c, st, KC_COMMIT);
    launch_commit(st, kv_view(kv), n_seqs, seq_slots, accept_len, blocks_in_use, c->pdl);
  }
  return check_cuda(c);
}

int hsd_verify_page(hsd_ctx* c, const hsd_kv* kv, int seq_slot, const int* pending_token, const int* draft_chunk,
                    int chunk_len, float log_tau, int* accept_len, int* emit_tokens, int* n_emit, int* row_argmax,
                    float* row_zmax, float* row_zdraft, void* workspace, size_t ws_bytes, void* cuda_stream) {
  if (!c || !pending_token || !accept_len || !emit_tokens || !n_emit) return HSD_ERR_INVALID_ARG;
  if (chunk_len < 0 || (chunk_len > 0 && !draft_chunk)) return HSD_ERR_INVALID_ARG;
  if (!(log_tau <= 0.f)) return HSD_ERR_INVALID_ARG;
  if (chunk_len + 1 > HSD_MAX_Q_LEN) return HSD_ERR_TOO_LONG;
  int rc = check_kv(kv);
  if (rc) return rc;
  if (seq_slot < 0 || seq_slot >= kv->n_slots) return HSD_ERR_INVALID_ARG;
  if ((long long)chunk_len + 1 > (long long)kv->max_blocks_per_seq * HSD_KV_BLOCK) return HSD_ERR_KV_CAPACITY;
  rc = check_ws(c, workspace, ws_bytes, chunk_len + 1, 1);
  if (rc) return rc;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  StepArgs a = {};
  a.n_seqs = 1; a.total_q = chunk_len + 1; a.max_q_len = chunk_len + 1; a.prefill = false;
  a.cu_q = nullptr; a.tokens = nullptr; a.pending = pending_token; a.draft = draft_chunk;
  a.seq_slots = nullptr; a.slot_base = seq_slot;
  return verify_common(c, kv, a, log_tau, accept_len, emit_tokens, n_emit, row_argmax, row_zmax, row_zdraft, workspace,
                       ws_bytes, st);
}

int hsd_kv_commit(hsd_ctx* c, const hsd_kv* kv, int n_seqs, const int* seq_slots, const int* accept_len,
                  int* blocks_in_use, void* cuda_stream) {
  if (!c || !accept_len || n_seqs <= 0) return HSD_ERR_INVALID_ARG;
  int rc = check_kv(kv);
  if (rc) return rc;
  if (!seq_slots && n_seqs > kv->n_slots) return HSD_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  Scope s(c, st, KC_COMMIT);
  launch_commit(st, kv_view(kv), n_seqs, seq_slots, accept_len, blocks_in_use, c->pdl);
  return check_cuda(c);
}

int hsd_verify_regions_host(hsd_ctx* c, const hsd_kv* kv, int n_seqs, const int* cu_q, const int* q_tokens,
                            const int* seq_slots, float log_tau, int commit, int* accept_len, int* emit_tokens,
                            int* n_emit, int* max_q_len_out, void* workspace, size_t ws_bytes, void* cuda_stream) {
  if (!c || !kv || !cu_q || !q_tokens || !accept_len || !emit_tokens || !n_emit || n_seqs <= 0) return HSD_ERR_INVALID_ARG;
  if (cu_q[0] != 0) return HSD_ERR_INVALID_ARG;
  int max_q = 0;
  for (int i = 0; i < n_seqs; ++i) {
    const int q = cu_q[i + 1] - cu_q[i];
    if (q <= 0) return HSD_ERR_INVALID_ARG;
    if (q > max_q) max_q = q;
  }
  const int total_q = cu_q[n_seqs];
  if (max_q > HSD_MAX_Q_LEN) return HSD_ERR_TOO_LONG;
  int rc = check_ws(c, workspace, ws_bytes, total_q, n_seqs);
  if (rc) return rc;
  const Ws w = carve(c, workspace, total_q, n_seqs);
  const size_t emit_ints = (size_t)n_seqs * max_q;
  const size_t out_ints = 2 * (size_t)n_seqs + emit_ints;
  if (out_ints > w.h_out_ints) return HSD_ERR_WORKSPACE;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);

  // pinned staging: [cu_q | q_tokens], from the next 16 bytes on [status words | accept_len | n_emit | emit_tokens]
  const size_t in_ints = (size_t)n_seqs + 1 + total_q, out_at = align_up(in_ints, 4);
  const size_t need = out_at + align_up(kStatusWords + out_ints, 4);
  if (need > c->pin_ints) {
    if (c->hg_exec) { cudaGraphExecDestroy(c->hg_exec); c->hg_exec = nullptr; }   // it names the old staging
    c->hg_seen_valid = false;
    if (c->pin) cudaFreeHost(c->pin);
    c->pin = nullptr;
    c->pin_ints = 0;
    if (cudaHostAlloc(reinterpret_cast<void**>(&c->pin), need * sizeof(int), cudaHostAllocDefault) != cudaSuccess)
      return fail_cuda(c);
    c->pin_ints = need;
  }
  int* p_cu = c->pin;
  int* p_tok = p_cu + n_seqs + 1;
  int* p_status = c->pin + out_at;
  int* p_acc = p_status + kStatusWords;
  int* p_nem = p_acc + n_seqs;
  int* p_emit = p_nem + n_seqs;
  memcpy(p_cu, cu_q, sizeof(int) * (n_seqs + 1));
  memcpy(p_tok, q_tokens, sizeof(int) * total_q);

  HostCallKey key;
  memset(&key, 0, sizeof(key));
  key.kv = *kv;
  key.seq_slots = seq_slots;
  key.workspace = workspace;
  key.ws_bytes = ws_bytes;
  key.stream = cuda_stream;
  key.n_seqs = n_seqs;
  key.total_q = total_q;
  key.max_q = max_q;
  key.commit = commit != 0;
  key.log_tau = log_tau;

  // the whole step on the stream: inputs in, verify (+ commit), results and status words out
  auto enqueue = [&]() -> int {
    {
      Scope s(c, st, KC_SETUP);
      launch_copy_words(st, w.h_in, c->pin, in_ints, false);   // (first of the call: nothing to overlap with)
    }
    int *accept = w.h_out, *n_em = accept + n_seqs, *emit = n_em + n_seqs;
    int r = hsd_verify_regions(c, kv, n_seqs, w.h_in, w.h_in + n_seqs + 1, seq_slots, max_q, total_q, log_tau, accept, emit,
                               n_em, nullptr, nullptr, nullptr, workspace, ws_bytes, cuda_stream);
    if (r) return r;
    if (commit) {
      r = hsd_kv_commit(c, kv, n_seqs, seq_slots, accept, nullptr, cuda_stream);
      if (r) return r;
    }
    {
      Scope s(c, st, KC_COMMIT);
      launch_copy_words(st, p_status, w.status, kStatusWords + out_ints, c->pdl);
    }
    return check_cuda(c);
  };

  const bool graph_stream = c->host_graph_ok && !c->profiling && st != nullptr && st != cudaStreamLegacy &&
                            st != cudaStreamPerThread;
  if (graph_stream && c->hg_exec && memcmp(&key, &c->hg_key, sizeof(key)) == 0) {
    if (cudaGraphLaunch(c->hg_exec, st) != cudaSuccess) return fail_cuda(c);
    c->launches += c->hg_launches;
  } else if (graph_stream && c->hg_seen_valid && memcmp(&key, &c->hg_seen, sizeof(key)) == 0) {
    // second call of this shape (the first one ran eagerly and set every one-time kernel attribute): capture it
    if (c->hg_exec) { cudaGraphExecDestroy(c->hg_exec); c->hg_exec = nullptr; }
    if (cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal) != cudaSuccess) return fail_cuda(c);
    const long long before = c->launches;
    rc = enqueue();
    cudaGraph_t graph = nullptr;
    const cudaError_t end = cudaStreamEndCapture(st, &graph);
    c->hg_launches = c->launches - before;
    c->launches = before;
    if (rc || end != cudaSuccess || !graph) {
      if (graph) cudaGraphDestroy(graph);
      c->hg_seen_valid = false;
      return rc ? rc : fail_cuda(c);
    }
    const cudaError_t inst = cudaGraphInstantiate(&c->hg_exec, graph, 0);
    cudaGraphDestroy(graph);
    if (inst != cudaSuccess) { c->hg_exec = nullptr; c->hg_seen_valid = false; return fail_cuda(c); }
    c->hg_key = key;
    if (cudaGraphLaunch(c->hg_exec, st) != cudaSuccess) return fail_cuda(c);
    c->launches += c->hg_launches;
  } else {
    rc = enqueue();
    if (rc) return rc;
    c->hg_seen = key;
    c->hg_seen_valid = true;
  }
  if (cudaStreamSynchronize(st) != cudaSuccess) return fail_cuda(c);
  memcpy(accept_len, p_acc, sizeof(int) * n_seqs);
  memcpy(n_emit, p_nem, sizeof(int) * n_seqs);
  memcpy(emit_tokens, p_emit, sizeof(int) * emit_ints);
  if (max_q_len_out) *max_q_len_out = max_q;
  return p_status[0] ? HSD_ERR_DEVICE_CHECK : HSD_OK;
}

int hsd_device_status(hsd_ctx* c, const void* workspace, void* cuda_stream, int status[4]) {
  if (!c || !workspace || !status) return HSD_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  if (cudaMemcpyAsync(status, workspace, 4 * sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return fail_cuda(c);
  return status[0] ? HSD_ERR_DEVICE_CHECK : HSD_OK;
}

int hsd_last_cuda_error(const hsd_ctx* c) { return c ? c->last_cuda_error : 0; }
long long hsd_launch_count(const hsd_ctx* c) { return c ? c->launches : 0; }

int hsd_profile_enable(hsd_ctx* c, int enable) {
  if (!c) return HSD_ERR_INVALID_ARG;
  for (auto& e : c->prof_events) { c->event_pool.push_back(e.a); c->event_pool.push_back(e.b); }
  c->prof_events.clear();
  memset(c->prof_ms, 0, sizeof(c->prof_ms));
  memset(c->prof_n, 0, sizeof(c->prof_n));
  c->profiling = enable != 0;
  return HSD_OK;
}

int hsd_profile_read(hsd_ctx* c, int cap, const char** names, double* total_ms, long long* launches) {
  if (!c || cap < 0) return HSD_ERR_INVALID_ARG;
  for (auto& e : c->prof_events) {
    float ms = 0.f;
    if (cudaEventSynchronize(e.b) != cudaSuccess || cudaEventElapsedTime(&ms, e.a, e.b) != cudaSuccess)
      return fail_cuda(c);
    c->prof_ms[e.kc] += ms;
    c->prof_n[e.kc] += 1;
  }
  for (auto& e : c->prof_events) {
    c->event_pool.push_back(e.a);
    c->event_pool.push_back(e.b);
  }
  c->prof_events.clear();
  int n = 0;
  for (int k = 0; k < KC_COUNT; ++k) {
    if (!c->prof_n[k]) continue;
    if (n < cap) {
      if (names) names[n] = kernel_class_name(k);
      if (total_ms) total_ms[n] = c->prof_ms[k];
      if (launches) launches[n] = c->prof_n[k];
    }
    ++n;
  }
  return n;
}

int hsd_debug_logits(hsd_ctx* c, const void* workspace, int total_q, int n_seqs, float* logits, void* cuda_stream) {
  if (!c || !workspace || !logits || total_q <= 0 || n_seqs <= 0) return HSD_ERR_INVALID_ARG;
  const Ws w = carve(c, const_cast<void*>(workspace), total_q, n_seqs);
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  Scope s(c, st, KC_DEBUG);
  GemmOut o = {logits, c->md.V, nullptr, nullptr, nullptr};
  launch_gemm_simt(st, w.h, c->lm_head, total_q, c->md.V, c->md.d, GM_STORE_F32, o);
  return check_cuda(c);
}

int hsd_debug_buffer(hsd_ctx* c, const void* workspace, int total_q, int n_seqs, const char* name, void** ptr,
                     size_t* bytes) {
  if (!c || !workspace || !name || !ptr || !bytes || total_q <= 0 || n_seqs <= 0) return HSD_ERR_INVALID_ARG;
  const Ws w = carve(c, const_cast<void*>(workspace), total_q, n_seqs);
  const ModelDims& md = c->md;
  const size_t T = (size_t)total_q;
  if (!strcmp(name, "x")) { *ptr = w.x; *bytes = 4 * T * md.d; }
  else if (!strcmp(name, "h")) { *ptr = w.h; *bytes = 2 * T * md.d; }
  else if (!strcmp(name, "q")) { *ptr = w.q; *bytes = 2 * T * md.Hq * md.D; }
  else if (!strcmp(name, "attn")) { *ptr = w.attn; *bytes = 2 * T * md.Hq * md.D; }
  else if (!strcmp(name, "act")) { *ptr = w.act; *bytes = 2 * T * md.ffn; }
  else return HSD_ERR_INVALID_ARG;
  return HSD_OK;
}

int hsd_debug_tap(hsd_ctx* c, int layer, int which, void* dst, size_t dst_bytes) {
  if (!c) return HSD_ERR_INVALID_ARG;
  if (layer < 0) { c->tap_layer = -1; return HSD_OK; }
  if (layer >= c->md.n_layers || which < HSD_TAP_X || which > HSD_TAP_X_MID || !dst) return HSD_ERR_INVALID_ARG;
  c->tap_layer = layer;
  c->tap_which = which;
  c->tap_dst = dst;
  c->tap_bytes = dst_bytes;
  return HSD_OK;
}

// Shared body of the LM-head operator: rows of h -> per-row argmax / max logit / next-token logit, with
// `best` (8 bytes per row) as the only scratch.
static int lm_head_argmax_impl(hsd_ctx* c, const void* h, int rows, const int* next_tokens, unsigned long long* best,
                               int* argmax, float* zmax, float* zdraft, cudaStream_t st) {
  const ModelDims& md = c->md;
  {
    Scope s(c, st, KC_LMHEAD);
    launch_clear_best(st, best, next_tokens ? zdraft : nullptr, rows, false);
  }
  {
    Scope s(c, st, KC_LMHEAD);
    GemmOut o = {nullptr, 0, best, zdraft, next_tokens};
    if (c->simt) {
      launch_gemm_simt(st, static_cast<const bf16*>(h), c->lm_head, rows, md.V, md.d, GM_ARGMAX, o);
    } else {
      GemmSm100Args g = {};
      if (make_tmap_2d(&g.tmA, h, rows, md.d, gemm_a_box_rows(rows))) return HSD_ERR_CUDA;
      g.tmB = &c->tm_lm_head;
      g.M = rows; g.n_out = md.V; g.K = md.d; g.mode = GS_ARGMAX;
      g.out = o;
      g.status = nullptr; g.n_sms = c->n_sms; g.max_splits = 1; g.pdl = false; g.pair = c->pair;
      g.tile = planned_tile(c, g, c->tiles_lm_head);
      if (launch_gemm_sm100(st, g)) return fail_cuda(c);
    }
  }
  {
    Scope s(c, st, KC_LMHEAD);
    launch_unpack_best(st, best, rows, argmax, zmax, false);
  }
  return check_cuda(c);
}

int hsd_op_lm_head_argmax(hsd_ctx* c, const void* h, int rows, const int* next_tokens, void* scratch,
                          size_t scratch_bytes, int* argmax, float* zmax, float* zdraft, void* cuda_stream) {
  if (!c || !h || !scratch || !argmax || !zmax || rows <= 0) return HSD_ERR_INVALID_ARG;
  if (next_tokens && !zdraft) return HSD_ERR_INVALID_ARG;
  if (scratch_bytes < (size_t)rows * 8 || (reinterpret_cast<uintptr_t>(scratch) & 7)) return HSD_ERR_WORKSPACE;
  return lm_head_argmax_impl(c, h, rows, next_tokens, static_cast<unsigned long long*>(scratch), argmax, zmax, zdraft,
                             static_cast<cudaStream_t>(cuda_stream));
}

// ---- the entry point for callers that cannot allocate device memory -------------------------------------
// Scratch of the no-allocation LM-head operator: one 8-byte running-best word per row.  The array lives in the
// library image, so every device that loads the library carries these 64 KB until the process exits.  In host
// code the symbol below is only a stand-in; the device address comes from cudaGetSymbolAddress.
static __device__ __align__(256) unsigned char g_noalloc_scratch[HSD_NOALLOC_MAX_ROWS * 8];
static unsigned long long* g_noalloc_addr[64] = {};   // per device ordinal, filled on that device's first call

int hsd_op_lm_head_argmax_noalloc(hsd_ctx* c, const void* h, int rows, const int* next_tokens, int* argmax,
                                  float* zmax, float* zdraft, void* cuda_stream) {
  if (!c || !h || !argmax || !zmax || rows <= 0) return HSD_ERR_INVALID_ARG;
  if (next_tokens && !zdraft) return HSD_ERR_INVALID_ARG;
  if (rows > HSD_NOALLOC_MAX_ROWS) return HSD_ERR_TOO_LONG;
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess) return fail_cuda(c);
  if (dev != c->device || dev < 0 || dev >= 64) return HSD_ERR_INVALID_ARG;
  if (!g_noalloc_addr[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return fail_cuda(c);
    g_noalloc_addr[dev] = static_cast<unsigned long long*>(p);
  }
  const bool was_profiling = c->profiling;   // event objects are created on demand while profiling: keep it off here
  c->profiling = false;
  const int rc = lm_head_argmax_impl(c, h, rows, next_tokens, g_noalloc_addr[dev], argmax, zmax, zdraft,
                                     static_cast<cudaStream_t>(cuda_stream));
  c->profiling = was_profiling;
  return rc;
}

int hsd_debug_set_gemm_tile(hsd_ctx* c, int tile_n, int k_slices) {
  if (!c || tile_n < 0 || k_slices < 0) return HSD_ERR_INVALID_ARG;
  c->force_bn = tile_n;
  c->force_splits = k_slices;
  return HSD_OK;
}

int hsd_debug_host_work(const hsd_ctx* c, long long* tile_choices, int* weight_maps, int* gemm_kernels) {
  if (!c || !tile_choices || !weight_maps || !gemm_kernels) return HSD_ERR_INVALID_ARG;
  *tile_choices = c->tile_choices;
  *weight_maps = c->n_weight_maps;
  *gemm_kernels = c->n_gemm_kernels;
  return HSD_OK;
}

int hsd_debug_tile(const hsd_ctx* c, int projection, int rows, int* out) {
  if (!c || c->simt || !out || projection < 0 || projection > 4 || rows < 1 || rows > TilePlan::kRows) return HSD_ERR_INVALID_ARG;
  const TilePlan* plans[5] = {&c->tiles_qkv, &c->tiles_o, &c->tiles_gate_up, &c->tiles_down, &c->tiles_lm_head};
  const TileChoice& t = plans[projection]->of[gemm_row_class(rows)];
  out[0] = t.bn; out[1] = t.splits; out[2] = t.pair;
  return HSD_OK;
}

int hsd_debug_set_attn_plan(hsd_ctx* c, int target_items, int min_kv_tiles) {
  if (!c || target_items < 0 || min_kv_tiles < 0) return HSD_ERR_INVALID_ARG;
  c->attn_target_items = target_items ? target_items : attn_grid(c);
  c->attn_min_chunk = min_kv_tiles ? 2 * min_kv_tiles : attn_min_chunk(c->md);
  c->attn_fine = min_kv_tiles != 0;
  return HSD_OK;
}

int hsd_op_linear(hsd_ctx* c, const void* A, const void* W, void* C, int M, int n_out, int K, int mode,
                  void* cuda_stream) {
  if (!c || !A || !W || !C || M <= 0 || n_out <= 0 || K <= 0) return HSD_ERR_INVALID_ARG;
  if (K % 64 || n_out % 64 || mode < 0 || mode > 2 || (mode == 2 && n_out % 128)) return HSD_ERR_SHAPE;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  const int ldc = mode == 2 ? n_out / 2 : n_out;
  Scope s(c, st, KC_DEBUG);
  if (c->simt) {
    GemmOut o = {C, ldc, nullptr, nullptr, nullptr};
    launch_gemm_simt(st, static_cast<const bf16*>(A), static_cast<const bf16*>(W), M, n_out, K, mode, o);
    return check_cuda(c);
  }
  GemmSm100Args g = {};
  WeightMaps wm;
  if (make_tmap_2d(&g.tmA, A, M, K, gemm_a_box_rows(M))) return HSD_ERR_CUDA;
  if (mode == 1 ? make_tmap_2d_f32(&g.tmC, C, M, ldc, 32) : make_tmap_2d(&g.tmC, C, M, ldc, 32)) return HSD_ERR_CUDA;
  g.tmB = &wm;
  g.M = M; g.n_out = n_out; g.K = K; g.mode = mode;
  g.out.C = C; g.out.ldc = ldc;
  g.status = nullptr; g.n_sms = c->n_sms; g.max_splits = c->max_splits; g.pdl = false; g.pair = c->pair;
  g.tile = choose_tile(c, g, c->force_bn, c->force_splits);
  int kernels = 0;
  if (gemm_sm100_prepare(mode, &kernels)) return fail_cuda(c);
  if (g.tile.bn && make_tmap_2d(&wm.half_tile(g.tile.bn), W, n_out, K, g.tile.bn / 2)) return HSD_ERR_CUDA;
  if (launch_gemm_sm100(st, g)) return fail_cuda(c);
  return check_cuda(c);
}

}  // extern "C"
