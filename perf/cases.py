"""What a user of the library has it do, as measurable cases: verification steps of every form (region batches, plain
decode, page chunks over long contexts, mixed serving batches, candidate trees, the host-buffer call) and the prefill
that comes before them, through the package's public entry points.

A case is a dict of plain values; the per-sequence lengths follow from its `shape_seed`, everything else (weights apart,
which belong to the model and not to a call) from the seed given to `prepare`: visual rows, token ids, drafts, agreement
lengths and the physical block placement.

The decoders' weights follow the recipe of `inputs.make_chain_weights` with branches strong enough (scale 0.05) that the
residual stream is mostly what the layers wrote: the logits carry every layer's arithmetic, and the emitted tokens are
still decided by wide margins, so that token outputs do not depend on a summation order."""
import math

import numpy as np
import torch

from paper_2602_12957_b200 import binding as B
from paper_2602_12957_b200 import inputs as I
from paper_2602_12957_b200 import roofline as RL
from paper_2602_12957_b200 import runtime as R

MODELS = {
    "tiny": I.TINY,
    "decoder": I.DECODER,
    # an 8-layer slice of the wider decoder with 128-wide heads, with the per-head q/k norm of such decoders
    "decoder_hd128": I.ModelConfig(n_layers=8, d_model=2048, n_heads=16, n_kv_heads=8, head_dim=128, d_ffn=8192, vocab=32768,
                                   qk_norm=True),
}
BRANCH_SCALE = 0.05
LOG_TAU = math.log(0.75)       # the paper's acceptance threshold (Sec. 4.3); 0 = exact greedy match
PROMPT = 16                    # the last rows of a prefix are text, as a prompt's are
WINDOW = 3                     # reference window of the matching (Sec. 4.3)
TREE_ROWS = 128
DRAFT_COPY = 320               # tokens of one pipeline draft in the tree steps
PREFILL_ROWS = 16384           # rows of one prefill call while a case's context is laid down


def listed():
    return [
        # one small decoder layer, four short regions: launches and latency are all there is
        dict(name="tiny_regions", kind="regions", model="tiny", seqs=4, prefix_lo=128, prefix_hi=128, draft_mean=16,
             draft_lo=16, draft_hi=16, pages=0, exact=True, shape_seed=1),
        # plain decoding: one row per sequence, no drafts (a step after nothing matched)
        dict(name="decode_16", kind="regions", model="decoder", seqs=16, prefix_lo=256, prefix_hi=1024, draft_mean=0,
             draft_lo=0, draft_hi=0, pages=0, exact=True, shape_seed=2),
        # short drafts of a region batch: the memory-bound regime
        dict(name="short_drafts", kind="regions", model="decoder", seqs=16, prefix_lo=256, prefix_hi=1024, draft_mean=8,
             draft_lo=8, draft_hi=8, pages=0, exact=True, shape_seed=3),
        # Stage 1 of a page: 16 regions with ragged drafts
        dict(name="regions", kind="regions", model="decoder", seqs=16, prefix_lo=256, prefix_hi=1024, draft_mean=64,
             draft_lo=8, draft_hi=256, pages=0, exact=True, shape_seed=4),
        # the same step for a caller whose drafts and results live in host memory
        dict(name="regions_host", kind="host", model="decoder", seqs=12, prefix_lo=200, prefix_hi=1500, draft_mean=40,
             draft_lo=4, draft_hi=160, pages=0, exact=True, shape_seed=5),
        # Stage 2 in its chunked form: one page chunk over the page's context
        dict(name="page_512", kind="page", model="decoder", context=7936, chunk=512, exact=True, shape_seed=6),
        # a long document's chunk over 16 k committed tokens
        dict(name="long_2048", kind="page", model="decoder", context=16384, chunk=2048, exact=True, shape_seed=7),
        # a serving batch: 64 regions of several pages and two page chunks in one call
        dict(name="mixed", kind="regions", model="decoder", seqs=64, prefix_lo=128, prefix_hi=2048, draft_mean=96,
             draft_lo=8, draft_hi=512, pages=2, exact=False, shape_seed=8),
        # Stage 1 with candidate trees: matching, tree step, compaction, 16 lanes
        dict(name="tree_16_lanes", kind="tree", model="decoder", lanes=16, prefix_lo=256, prefix_hi=1024, drafts=2,
             exact=False, shape_seed=9),
        # Stage 2 with candidate trees: one lane over the page's context, matched against every region's text
        dict(name="tree_1_lane", kind="tree", model="decoder", lanes=1, prefix_lo=4700, prefix_hi=4700, drafts=16,
             exact=False, shape_seed=10),
        # prefill of a page's region crops (visual rows, then a prompt)
        dict(name="prefill_crops", kind="prefill", model="decoder", seqs=16, prefix_lo=256, prefix_hi=1024, shape_seed=11),
        # the region step on the wider decoder with 128-wide heads and q/k norm
        dict(name="regions_hd128", kind="regions", model="decoder_hd128", seqs=16, prefix_lo=256, prefix_hi=1024,
             draft_mean=64, draft_lo=8, draft_hi=256, pages=0, exact=True, shape_seed=12),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: every kind of call, sizes spread over their logarithm, odd ones among them."""
    kind = rng.choice(["regions", "regions", "regions", "decode", "host", "page", "page", "tree", "prefill"])
    shape_seed = rng.randrange(1 << 30)
    model = rng.choice(["decoder", "decoder", "decoder", "decoder", "decoder_hd128", "tiny"])
    exact = rng.random() < 0.5
    prefix_lo = _log_int(rng, 64, 1024)
    prefix_hi = min(2048, prefix_lo + _log_int(rng, 1, 1024))
    if kind == "page":
        return dict(kind="page", model=model if model != "tiny" else "decoder", context=_log_int(rng, 500, 16384),
                    chunk=_log_int(rng, 16, 2048), exact=exact, shape_seed=shape_seed)
    if kind == "tree":
        return dict(kind="tree", model=model, lanes=_log_int(rng, 1, 16), prefix_lo=prefix_lo, prefix_hi=prefix_hi,
                    drafts=rng.choice([1, 2, 3, 5]), exact=exact, shape_seed=shape_seed)
    if kind == "prefill":
        return dict(kind="prefill", model=model, seqs=_log_int(rng, 1, 10), prefix_lo=prefix_lo,
                    prefix_hi=max(prefix_lo, min(1024, prefix_hi)), shape_seed=shape_seed)
    if kind == "decode":
        return dict(kind="regions", model=model, seqs=_log_int(rng, 1, 64), prefix_lo=prefix_lo, prefix_hi=prefix_hi,
                    draft_mean=0, draft_lo=0, draft_hi=0, pages=0, exact=exact, shape_seed=shape_seed)
    mean = _log_int(rng, 4, 128)
    return dict(kind=kind, model=model, seqs=_log_int(rng, 1, 40), prefix_lo=prefix_lo, prefix_hi=prefix_hi, draft_mean=mean,
                draft_lo=max(1, mean // 8), draft_hi=4 * mean, pages=1 if kind == "regions" and rng.random() < 0.15 else 0,
                exact=exact, shape_seed=shape_seed)


# ------------------------------------------------------------------------------------------------ shapes and work
def _shapes(case):
    """(committed rows, query rows) of every sequence of the call; a prefill starts from empty caches."""
    rng = np.random.Generator(np.random.PCG64(case["shape_seed"]))
    if case["kind"] == "page":
        return [case["context"]], [case["chunk"] + 1]
    n = case["lanes"] if case["kind"] == "tree" else case["seqs"]
    prefix = [int(v) for v in rng.integers(case["prefix_lo"], case["prefix_hi"] + 1, size=n)]
    if case["kind"] == "prefill":
        return [0] * n, prefix
    if case["kind"] == "tree":
        return prefix, [TREE_ROWS] * n
    if case["draft_hi"] == 0:
        draft = [0] * n
    else:
        draft = [int(v) for v in I.lognormal_lengths(rng, n, float(case["draft_mean"]), case["draft_lo"], case["draft_hi"])]
    for _ in range(case["pages"]):
        prefix.append(4352)
        draft.append(1024)
    return prefix, [k + 1 for k in draft]


def work(case):
    cfg = MODELS[case["model"]]
    context, q = _shapes(case)
    w = RL.step_work(cfg, context, q)
    if case["kind"] == "prefill":        # the LM head is needed for the last row of every sequence only
        head = 2.0 * cfg.vocab * cfg.d_model
        return {"bytes": w.bytes, "flops": w.flops - head * (sum(q) - len(q))}
    if case["kind"] == "tree":           # a node sees the context, itself and its ancestors: count the context and itself
        pairs = sum(r * (L + 1) for L, r in zip(context, q))
        return {"bytes": w.bytes, "flops": w.gemm_flops + 4.0 * cfg.n_heads * cfg.head_dim * cfg.n_layers * pairs}
    return {"bytes": w.bytes, "flops": w.flops}


def tolerance(case):
    # bf16 activations through up to 24 layers.  K slices add into the residual in arrival order, so the same call, made
    # twice, differs from itself: measured up to rel 3e-3, and 0.053 of the root mean square for single values; about
    # four times that.  Tokens and lengths are decided by margins far beyond it.
    return {"rel": 1.2e-2, "max": 0.2, "differ": 0.0}


# ------------------------------------------------------------------------------------------------ the models
_models = {}


def _model(name):
    """The decoder, its weights on the device and the order of its greedy text; made once, as a user's program does."""
    if name not in _models:
        cfg = MODELS[name]
        g = torch.Generator(device="cuda").manual_seed(I.BASE_SEED)
        d, f, hd = cfg.d_model, cfg.d_ffn, cfg.head_dim

        def normal(*shape, std=0.02, mean=0.0):
            return (torch.randn(*shape, generator=g, device="cuda") * std + mean).to(torch.bfloat16).float()

        layers = []
        for _ in range(cfg.n_layers):
            lw = {"attn_norm": normal(d, mean=1.0), "w_qkv": normal(cfg.qkv_out, d),
                  "w_o": normal(d, cfg.n_heads * hd) * BRANCH_SCALE, "ffn_norm": normal(d, mean=1.0),
                  "w_gate_up": normal(2 * f, d), "w_down": normal(d, f) * BRANCH_SCALE}
            if cfg.qk_norm:
                lw["q_norm"], lw["k_norm"] = normal(hd, std=0.1, mean=1.0), normal(hd, std=0.1, mean=1.0)
            layers.append({k: v.cpu().numpy() for k, v in lw.items()})
        embed = normal(cfg.vocab, d)
        order = torch.randperm(cfg.vocab, generator=g, device="cuda")
        lm_head = torch.empty_like(embed)
        lm_head[torch.roll(order, -1)] = embed[order] * 4.0        # order[i + 1] follows order[i]
        weights = {"layers": layers, "embed": embed.cpu().numpy(), "final_norm": normal(d, mean=1.0).cpu().numpy(),
                   "lm_head": lm_head.cpu().numpy()}
        place = torch.empty_like(order)
        place[order] = torch.arange(cfg.vocab, device="cuda")
        _models[name] = (R.DeviceModel(cfg, weights), order.cpu().numpy(), place.cpu().numpy())
    return _models[name]


# ------------------------------------------------------------------------------------------------ inputs
class State:
    """One engine with its cache, the call's inputs and its output buffers."""


def _i32(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).cuda()


def _prefix_inputs(cfg, lens, rng, seed):
    """Visual rows N(0, 1), then PROMPT token ids (a quarter of a very short prefix)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    rows = sum(lens)
    embeds = torch.randn(rows, cfg.d_model, generator=g, device="cuda").to(torch.bfloat16)
    ids = np.full(rows, -1, np.int32)
    at = 0
    for n in lens:
        k = max(1, min(PROMPT, n // 4))
        ids[at + n - k:at + n] = rng.integers(0, cfg.vocab, size=k)
        at += n
    return embeds, ids


def _prefill(model, kv, engine, lens, slots, embeds, ids, first):
    cu = np.concatenate([[0], np.cumsum(lens)])
    st = B.hsd_prefill(model.ctx, kv.c, len(lens), _i32(cu), embeds, _i32(ids), _i32(slots), int(cu[-1]), int(max(lens)), first,
                       engine.ws.ptr, engine.ws.bytes, torch.cuda.current_stream().cuda_stream)
    B.check(st, "hsd_prefill")


def _lay_down_context(model, kv, lens, rng, seed):
    """Fills the caches of slots 0.. with prefixes of the given lengths, in calls of at most PREFILL_ROWS rows."""
    first = torch.empty(len(lens), dtype=torch.int32, device="cuda")
    groups, rows = [[]], 0
    for i, n in enumerate(lens):
        if groups[-1] and rows + n > PREFILL_ROWS:
            groups.append([])
            rows = 0
        groups[-1].append(i)
        rows += n
    engine = R.Engine(model, kv, max(sum(lens[i] for i in g) for g in groups), max(len(g) for g in groups))
    for k, group in enumerate(groups):
        part = [lens[i] for i in group]
        embeds, ids = _prefix_inputs(model.cfg, part, rng, seed * 1000 + k)
        _prefill(model, kv, engine, part, group, embeds, ids, first[group[0]:group[-1] + 1])


def _walk(order, place, token, n):
    """The n tokens the decoder emits after `token`."""
    return order[(place[token] + 1 + np.arange(n)) % len(order)]


def prepare(case, seed):
    s = State()
    s.case = case
    model, order, place = _model(case["model"])
    cfg = model.cfg
    context, q = _shapes(case)
    rng = np.random.Generator(np.random.PCG64([case["shape_seed"], seed]))
    s.log_tau = 0.0 if case.get("exact", True) else LOG_TAU
    spare = TREE_ROWS if case["kind"] == "tree" else 0
    s.model = model.sibling(0) if case["kind"] == "host" else model      # (a context keeps the graph of one host call shape)
    s.kv = R.KvCache(s.model, [L + n + spare for L, n in zip(context, q)], seed=seed)
    total, longest = sum(q), max(q)

    if case["kind"] == "prefill":
        s.engine = R.Engine(s.model, s.kv, total, len(q))
        s.embeds, ids = _prefix_inputs(cfg, q, rng, seed)
        s.ids, s.cu = _i32(ids), _i32(np.concatenate([[0], np.cumsum(q)]))
        s.first = torch.zeros(len(q), dtype=torch.int32, device="cuda")
        s.rows, s.longest = total, longest
        return s

    _lay_down_context(s.model, s.kv, context, rng, seed)
    s.engine = R.Engine(s.model, s.kv, 2 * total if case["kind"] == "tree" else total, len(q))
    s.lens0 = s.kv.seq_lens.clone()
    s.out = {k: torch.zeros_like(v) for k, v in s.engine.alloc_outputs(len(q), longest, total).items()}

    if case["kind"] == "tree":
        # the pipeline's drafts: copies of the text with a wrong token every 16 on average, the window somewhere in it
        tokens, offsets, owners, windows = [], [0], [0], []
        for _ in range(case["lanes"]):
            text = _walk(order, place, int(rng.integers(0, cfg.vocab)), DRAFT_COPY)
            at = int(rng.integers(0, DRAFT_COPY - TREE_ROWS))
            windows.append(text[at:at + WINDOW])
            for k in range(case["drafts"]):
                copy = text.copy()
                wrong = rng.random(DRAFT_COPY) < 1.0 / 16
                if k == 0:
                    wrong[at:at + WINDOW] = False
                copy[wrong] = rng.integers(0, cfg.vocab, size=int(wrong.sum()))
                tokens.append(copy)
                offsets.append(offsets[-1] + DRAFT_COPY)
            owners.append(len(offsets) - 1)
        s.window = _i32(np.stack(windows))
        s.drafts, s.offsets, s.owners = _i32(np.concatenate(tokens)), _i32(offsets), _i32(owners)
        zeros = lambda *shape: torch.zeros(*shape, dtype=torch.int32, device="cuda")  # noqa: E731
        s.tree = {"q_tokens": zeros(total), "parent": zeros(total), "cu_q": zeros(len(q) + 1), "n_rows": zeros(len(q))}
        s.out["accept_rows"] = zeros(len(q), longest)
        s.out["row_zchild"] = s.out.pop("row_zdraft")
        s.rows = total
        return s

    # drafts that agree with the decoder's own text for a while; a page draft comes back to it after the wrong token
    pending, drafts = [], []
    for i, n in enumerate(q):
        k = n - 1
        p = int(rng.integers(0, cfg.vocab))
        agree = k if rng.random() < 0.5 else int(rng.uniform(0.2, 1.0) * k)
        drafts.append(I.plant_draft(_walk(order, place, p, k), k, agree, rng.integers(0, cfg.vocab, size=k), cfg.vocab,
                                    case["kind"] == "page" or i >= case.get("seqs", 0)))
        pending.append(p)
    tokens, cu = I.pack_queries(pending, drafts)
    s.longest, s.rows = longest, total
    if case["kind"] == "page":
        s.pending, s.chunk = _i32(tokens[:1]), _i32(tokens[1:])
    elif case["kind"] == "host":
        s.cu, s.tokens = torch.from_numpy(cu).pin_memory(), torch.from_numpy(tokens).pin_memory()
        s.stream = torch.cuda.Stream()
        s.stream.wait_stream(torch.cuda.current_stream())
        s.host_out = [torch.zeros(*n, dtype=torch.int32).pin_memory() for n in ((len(q),), (len(q), longest), (len(q),))]
    else:
        s.cu, s.tokens = _i32(cu), _i32(tokens)
    return s


def run(s):
    kind = s.case["kind"]
    pools = {"k_pool": s.kv.k_pool, "v_pool": s.kv.v_pool, "seq_lens": s.kv.seq_lens}
    if kind == "prefill":
        s.kv.seq_lens.zero_()                        # the caches of new crops
        st = B.hsd_prefill(s.model.ctx, s.kv.c, s.cu.numel() - 1, s.cu, s.embeds, s.ids, None, s.rows, s.longest, s.first,
                           s.engine.ws.ptr, s.engine.ws.bytes, torch.cuda.current_stream().cuda_stream)
        B.check(st, "hsd_prefill")
        return dict(pools, first_token=s.first)
    if kind == "host":
        accept, emit, n_emit = s.host_out
        with torch.cuda.stream(s.stream):
            s.kv.seq_lens.copy_(s.lens0)             # the step starts from the same committed lengths every time
            st, _ = B.hsd_verify_regions_host(s.model.ctx, s.kv.c, len(accept), s.cu, s.tokens, None, s.log_tau, 1, accept, emit,
                                              n_emit, s.engine.ws.ptr, s.engine.ws.bytes, s.stream.cuda_stream)
        B.check(st, "hsd_verify_regions_host")
        # (a row of emit_tokens is written up to its sequence's n_emit)
        emitted = np.where(np.arange(s.longest) < n_emit.numpy()[:, None], emit.numpy(), -1)
        return dict(pools, accept_len=accept.numpy(), n_emit=n_emit.numpy(), emitted=emitted)
    s.kv.seq_lens.copy_(s.lens0)
    if kind == "tree":
        s.engine.dsv_build(s.window, s.drafts, s.offsets, s.owners, TREE_ROWS, out=s.tree)
        out = s.engine.verify_tree(s.tree["q_tokens"], s.tree["cu_q"], s.tree["parent"], TREE_ROWS, s.rows, out=s.out,
                                   log_tau=s.log_tau)
        s.engine.commit_tree(out["accept_len"], out["accept_rows"])
        return dict(pools, tree=s.tree, **out)
    if kind == "page":
        out = s.engine.verify_page(0, s.pending, s.chunk, out=s.out, log_tau=s.log_tau)
    else:
        out = s.engine.verify_regions(s.tokens, s.cu, s.longest, s.rows, out=s.out, log_tau=s.log_tau)
    s.engine.commit(out["accept_len"])
    return dict(pools, **out)
