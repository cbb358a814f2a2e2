"""Attention over every form of plan against a float64 softmax of the same bf16 queries, keys and values: the context lengths
where the number of slices of a q-tile changes (8 KV blocks stay whole, heads of 128: 10; 12 are cut in two, 24 in three, 25 in
five, a long context in a square root's worth), slices as short as they come (4, 5, 7 and more of a q-tile: the combining pass takes three at a
time), whole ranges, and equal shares of the line with a q-tile cut across several shares.  Keys are spread widely enough that
a q-tile's slices differ in maximum and sum."""
import numpy as np
import pytest

from paper_2602_12957_b200 import inputs as I
from . import harness as H

pytestmark = pytest.mark.gpu

MODELS = {
    "tiny": (I.TINY, 8.0),                                      # one query head per kv head; key deviation
    "gqa": (I.ModelConfig(n_layers=1, d_model=1024, n_heads=16, n_kv_heads=8, head_dim=64, d_ffn=1024, vocab=4096), 4.0),
    "hd128": (I.ModelConfig(n_layers=1, d_model=2048, n_heads=16, n_kv_heads=8, head_dim=128, d_ffn=1024, vocab=4096,
                            qk_norm=True), 2.5),
}


@pytest.fixture(scope="module", params=list(MODELS))
def models(request):
    from paper_2602_12957_b200 import binding as B
    from paper_2602_12957_b200 import runtime as R
    cfg, spread = MODELS[request.param]
    model = R.DeviceModel(cfg, I.make_weights(cfg, 1))
    return {"cut": model, "whole": model.sibling(B.HSD_FLAG_DETERMINISTIC), "spread": spread}


def _check(model, spread, blocks, rows, plan):
    """One call with q-tiles of the given KV blocks; returns the plan's number of shares."""
    import torch
    from paper_2602_12957_b200 import binding as B
    from paper_2602_12957_b200 import runtime as R
    cfg, S = model.cfg, len(blocks)
    lens = [64 * b - rows if 64 * b > rows else 1 for b in blocks]       # the call's last row is its last block's last key
    kv = R.KvCache(model, [n + rows for n in lens])
    g = torch.Generator(device="cuda").manual_seed(7)
    kv.k_pool.copy_(torch.randn(kv.k_pool.shape, generator=g, device="cuda") * spread)
    kv.v_pool.copy_(torch.randn(kv.v_pool.shape, generator=g, device="cuda"))
    eng = R.Engine(model, kv, rows * S, S)
    toks = eng._i32(np.random.default_rng(rows + sum(blocks)).integers(0, cfg.vocab, rows * S))
    try:
        B.check(B.hsd_debug_set_attn_plan(model.ctx, *plan))
        q, out = H.layer0_attention(eng, toks, eng._i32(np.arange(S + 1) * rows), lens, [rows] * S)
    finally:
        B.hsd_debug_set_attn_plan(model.ctx, 0, 0)
    want, spread_out = H.attention_float64(cfg, kv, q, lens, [rows] * S)
    over = (out.double() - want).abs() / H.attention_tolerance(want, spread_out)
    assert float(over.max()) <= 1, float(over.max())
    off = eng.ws.ptr - eng.ws._raw.data_ptr()
    return int(eng.ws._raw[off:off + 64].view(torch.int32)[5])           # status word 5: shares per kv head


def _tiles(cfg, blocks, rows):
    """KV blocks of every q-tile of the call."""
    per = 128 * cfg.n_kv_heads // cfg.n_heads
    return [((64 * b - rows if 64 * b > rows else 1) + min(rows, t + per) + 63) // 64 for b in blocks for t in range(0, rows, per)]


@pytest.mark.parametrize("blocks", [[1], [8], [9], [12, 13], [18, 19], [24], [25], [8, 9, 24, 25, 3], [200]])
@pytest.mark.parametrize("rows", [1, 20, 65])
def test_slices(models, blocks, rows):
    _check(models["cut"], models["spread"], blocks, rows, (0, 0))


@pytest.mark.parametrize("blocks", [[8], [10], [14], [7, 9, 3], [24, 25], [200]])
@pytest.mark.parametrize("rows", [1, 20, 65])
def test_slices_of_two_blocks(models, blocks, rows):
    shares = _check(models["cut"], models["spread"], blocks, rows, (1 << 20, 1))
    slices = sum((n + 1) // 2 for n in _tiles(models["cut"].cfg, blocks, rows))
    assert shares == slices if slices <= 16 else shares > 8


@pytest.mark.parametrize("blocks", [[9], [24, 25], [200]])
@pytest.mark.parametrize("rows", [1, 65])
def test_whole(models, blocks, rows):
    shares = _check(models["whole"], models["spread"], blocks, rows, (0, 0))
    assert shares == len(_tiles(models["whole"].cfg, blocks, rows))


@pytest.mark.parametrize("finest", [0, 1])
@pytest.mark.parametrize("blocks", [[60, 3, 3, 3, 3, 3], [3, 40, 2, 2, 30], [150] + [3] * 12])
def test_line(models, blocks, finest):
    # one share fewer than q-tiles: the ranges are laid end to end, and the long ones cut across three to nine shares
    shares = _check(models["cut"], models["spread"], blocks, 20, ((len(blocks) - 1) * models["cut"].cfg.n_kv_heads, finest))
    assert shares == len(blocks) - 1
