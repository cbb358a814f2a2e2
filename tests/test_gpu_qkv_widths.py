"""The QKV projection with its rotary epilogue and K/V stores on every tile width (192 columns are three heads, and the last tile
of 32 heads has one too many; pairs too): queries and K/V rows equal the narrowest tile's bit by bit, as K is summed in one order.
And the width that a step of wide heads takes, whose epilogue is dear."""
import numpy as np
import pytest

from paper_2602_12957_b200 import inputs as I

from . import harness as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("head_dim", [64, 128])
@pytest.mark.parametrize("qk_norm", [False, True])
@pytest.mark.parametrize("rows", [[1], [65, 40], [130, 127, 3]])
def test_widths_agree(rows, qk_norm, head_dim):
    import torch
    from paper_2602_12957_b200 import binding as B
    from paper_2602_12957_b200 import runtime as R
    cfg = I.ModelConfig(n_layers=1, d_model=1024, n_heads=16, n_kv_heads=8, head_dim=head_dim, d_ffn=1024, vocab=4096, qk_norm=qk_norm)
    model = R.DeviceModel(cfg, I.make_weights(cfg, 2), B.HSD_FLAG_DETERMINISTIC)
    S, T = len(rows), sum(rows)
    lens = [70] * S
    toks = np.random.default_rng(T).integers(0, cfg.vocab, T)
    got = {}
    try:
        tiles = (64, 128, 192, 256, 384, 448, 512) if head_dim == 64 else (128, 256, 384, 512)
        for tile in tiles:
            kv = R.KvCache(model, [70 + n for n in rows], seed=3)
            kv.k_pool.zero_()
            kv.v_pool.zero_()
            eng = R.Engine(model, kv, T, S)
            B.check(B.hsd_debug_set_gemm_tile(model.ctx, tile, 0))
            q, _ = H.layer0_attention(eng, eng._i32(toks), eng._i32(np.concatenate([[0], np.cumsum(rows)])), lens, rows)
            got[tile] = (q.clone(), kv.k_pool.clone(), kv.v_pool.clone())
    finally:
        B.hsd_debug_set_gemm_tile(model.ctx, 0, 0)
    first = got[tiles[0]]
    assert float(first[1].abs().max()) > 0 and float(first[2].abs().max()) > 0
    for tile, out in got.items():
        assert all(torch.equal(a, b) for a, b in zip(out, first)), tile


def test_wide_heads_take_narrow_tiles():
    from paper_2602_12957_b200 import binding as B
    from paper_2602_12957_b200 import runtime as R
    cfg = I.ModelConfig(n_layers=1, d_model=2048, n_heads=16, n_kv_heads=8, head_dim=128, d_ffn=8192, vocab=4096, qk_norm=True)
    model = R.DeviceModel(cfg, I.make_weights(cfg, 2))
    for rows in (513, 612, 640, 700, 768):
        # the rotary epilogue of 128-column heads: 121 us a layer of 612 rows on 256-wide tiles, 112 on these
        assert B.hsd_debug_tile(model.ctx, 0, rows) == (B.HSD_OK, (128, 1, 1)), rows
    for rows in (305, 612):      # gate/up: 88.8 us a layer of 305 rows on single tiles, 85.9 on pairs; 121 and 117 of 612 rows
        assert B.hsd_debug_tile(model.ctx, 2, rows) == (B.HSD_OK, (224, 1, 1)), rows
    assert B.hsd_debug_tile(model.ctx, 5, 1)[0] == B.hsd_debug_tile(model.ctx, 0, 8193)[0] == B.HSD_ERR_INVALID_ARG
