"""RMSNorm at the row counts where its rows per CTA change: with 148 SMs from 589 rows on for the launch that also gathers the
set-up's verdicts (the first of a step), from 593 for the others, and around a CTA's rows; against float64 of the same inputs."""
import numpy as np
import pytest

from paper_2602_12957_b200 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [1, 3, 4, 5, 8, 9, 587, 588, 589, 592, 593, 597])
def test_norm_rows(rows):
    import torch
    from paper_2602_12957_b200 import binding as B
    from paper_2602_12957_b200 import runtime as R
    cfg = I.ModelConfig(n_layers=1, d_model=256, n_heads=4, n_kv_heads=2, head_dim=64, d_ffn=256, vocab=1024)
    weights = I.make_weights(cfg, 4)
    rng = np.random.default_rng(rows)
    for lw in weights["layers"]:
        lw["attn_norm"], lw["ffn_norm"] = (I.bf16_round(1.0 + 0.3 * rng.standard_normal(cfg.d_model, dtype=np.float32)) for _ in range(2))
    model = R.DeviceModel(cfg, weights, B.HSD_FLAG_DETERMINISTIC)
    eng = R.Engine(model, R.KvCache(model, [rows]), rows, 1)
    toks, cu = eng._i32(rng.integers(0, cfg.vocab, rows)), eng._i32([0, rows])
    got = {}
    for which, dtype in ((B.HSD_TAP_H_ATTN, torch.bfloat16), (B.HSD_TAP_X_MID, torch.float32), (B.HSD_TAP_H_FFN, torch.bfloat16)):
        out = torch.full((rows, cfg.d_model), 7.0, dtype=dtype, device=model.device)
        B.check(B.hsd_debug_tap(model.ctx, 0, which, out, out.numel() * out.element_size()))
        eng.verify_regions(toks, cu, rows, rows)
        eng.check_device("verify_regions")
        got[which] = out.double()
    embed = model.embed[toks.long()].double()
    for x, h, gain in ((embed, got[B.HSD_TAP_H_ATTN], "attn_norm"), (got[B.HSD_TAP_X_MID], got[B.HSD_TAP_H_FFN], "ffn_norm")):
        want = x / torch.sqrt((x * x).mean(1, keepdim=True) + cfg.rms_eps) * model.layers[0][gain].double()
        # one rounding to bf16, whose 8 significant bits are off by half a unit of the last, at most 2^-8 of the value; the fp32
        # sums and products before it by ~2^-20 (d additions, their errors' signs mixed)
        assert bool(((h - want).abs() <= (2.0 ** -8 + 2.0 ** -18) * want.abs()).all()), gain
