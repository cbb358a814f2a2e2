"""The QKV projection with its rotary epilogue and K/V stores on every tile width (192 columns are three heads, and the last tile
of 32 heads has one too many; pairs too): queries and K/V rows equal the 64-wide tile's bit by bit, as K is summed in one order."""
import numpy as np
import pytest

from paper_2602_12957_b200 import inputs as I

from . import harness as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("qk_norm", [False, True])
@pytest.mark.parametrize("rows", [[1], [65, 40], [130, 127, 3]])
def test_widths_agree(rows, qk_norm):
    import torch
    from paper_2602_12957_b200 import binding as B
    from paper_2602_12957_b200 import runtime as R
    cfg = I.ModelConfig(n_layers=1, d_model=1024, n_heads=16, n_kv_heads=8, head_dim=64, d_ffn=1024, vocab=4096, qk_norm=qk_norm)
    model = R.DeviceModel(cfg, I.make_weights(cfg, 2), B.HSD_FLAG_DETERMINISTIC)
    S, T = len(rows), sum(rows)
    lens = [70] * S
    toks = np.random.default_rng(T).integers(0, cfg.vocab, T)
    got = {}
    try:
        for tile in (64, 128, 192, 256, 384, 448, 512):
            kv = R.KvCache(model, [70 + n for n in rows], seed=3)
            kv.k_pool.zero_()
            kv.v_pool.zero_()
            eng = R.Engine(model, kv, T, S)
            B.check(B.hsd_debug_set_gemm_tile(model.ctx, tile, 0))
            q, _ = H.layer0_attention(eng, eng._i32(toks), eng._i32(np.concatenate([[0], np.cumsum(rows)])), lens, rows)
            got[tile] = (q.clone(), kv.k_pool.clone(), kv.v_pool.clone())
    finally:
        B.hsd_debug_set_gemm_tile(model.ctx, 0, 0)
    assert float(got[64][1].abs().max()) > 0 and float(got[64][2].abs().max()) > 0
    for tile, out in got.items():
        assert all(torch.equal(a, b) for a, b in zip(out, got[64])), tile
