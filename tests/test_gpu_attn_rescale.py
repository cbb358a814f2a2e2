"""Attention where later scores outgrow the exponent reference (the maximum of the first 64 keys a row saw): keys planted along
single rows' queries lift those rows, and only those rows of a warp, by 50 to 150 binary orders, in the second block, in the
middle, behind a slice's border, and several times within one item; against a float64 softmax."""
import math

import numpy as np
import pytest

from paper_2602_12957_b200 import inputs as I
from . import harness as H
from .test_gpu_attn_slices import models  # noqa: F401  (the three decoders)

pytestmark = pytest.mark.gpu

ROWS, BLOCKS = 20, [14, 30]
# row -> (key, binary orders above the rest) of the keys planted along its query
PLANT = {0: [(64, 50), (200, 100), (9 * 64 + 5, 150)], 3: [(6 * 64 + 63, 60)], 9: [(8 * 64, 60)], 12: [(70, 45), (71, 52)],
         19: [(4 * 64 + 1, 55), (12 * 64 + 9, 110)]}


@pytest.mark.parametrize("plan", ["whole", "default", "two blocks", "line"])
def test_scores_outgrow_the_reference(models, plan):  # noqa: F811
    import torch
    from paper_2602_12957_b200 import binding as B
    from paper_2602_12957_b200 import runtime as R
    model = models["whole" if plan == "whole" else "cut"]
    cfg, S = model.cfg, len(BLOCKS)
    group, sc = cfg.n_heads // cfg.n_kv_heads, math.log2(math.e) / math.sqrt(cfg.head_dim)
    lens = [64 * b - ROWS for b in BLOCKS]
    kv = R.KvCache(model, [n + ROWS for n in lens])
    g = torch.Generator(device="cuda").manual_seed(7)
    kv.k_pool.copy_(torch.randn(kv.k_pool.shape, generator=g, device="cuda") * 0.5)
    kv.v_pool.copy_(torch.randn(kv.v_pool.shape, generator=g, device="cuda"))
    eng = R.Engine(model, kv, ROWS * S, S)
    toks = eng._i32(np.random.default_rng(5).integers(0, cfg.vocab, ROWS * S))
    cu = eng._i32(np.arange(S + 1) * ROWS)
    q, _ = H.layer0_attention(eng, toks, cu, lens, [ROWS] * S)      # (the queries do not depend on the cache)
    for s in range(S):
        for row, keys in PLANT.items():
            for key, orders in keys:
                for h in range(cfg.n_kv_heads):
                    along = q[s * ROWS + row].view(cfg.n_heads, -1)[h * group + row % group].float()
                    kv.k_pool[0, kv.block_table[s, key // 64], h, key % 64] = along * (orders / (sc * float(along @ along)))
    try:
        B.check(B.hsd_debug_set_attn_plan(model.ctx, *{"two blocks": (1 << 20, 1), "line": (cfg.n_kv_heads, 0)}.get(plan, (0, 0))))
        q, out = H.layer0_attention(eng, toks, cu, lens, [ROWS] * S)
    finally:
        B.hsd_debug_set_attn_plan(model.ctx, 0, 0)
    want, spread = H.attention_float64(cfg, kv, q, lens, [ROWS] * S)
    over = (out.double() - want).abs() / H.attention_tolerance(want, spread)
    assert float(over.max()) <= 1, float(over.max())
    # the inputs do what they are for: of the first sequence's rows some outgrow their reference by more than the 40 orders
    # that make the library take a new one, others (of the same warp) stay far below
    k = kv.k_pool[0][kv.block_table[0, :BLOCKS[0]].long()].permute(1, 0, 2, 3).reshape(cfg.n_kv_heads, -1, cfg.head_dim).double()
    z = torch.stack([q[:ROWS].view(ROWS, cfg.n_heads, -1)[:, h].double() @ k[h // group, :lens[0]].T for h in range(cfg.n_heads)]) * sc
    grown = z.amax(2) - z[:, :, :64].amax(2)
    assert bool(((grown > 42).sum(1) >= 1).all()) and bool(((grown < 36).sum(1) >= 4).all())
