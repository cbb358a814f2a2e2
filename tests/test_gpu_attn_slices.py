"""Attention at the context lengths where the number of slices of a q-tile changes (8 KV blocks stay whole, 9 are cut in two,
up to 24 in three, a long context in a square root's worth), against a context that never cuts a KV range."""
import numpy as np
import pytest

from paper_2602_12957_b200 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("blocks", [[1], [8], [9], [12, 13], [18, 19], [24], [25], [8, 9, 24, 25, 3], [200]])
@pytest.mark.parametrize("rows", [1, 20, 65])
def test_slices(blocks, rows):
    import torch
    from paper_2602_12957_b200 import binding as B
    from paper_2602_12957_b200 import runtime as R
    weights = I.make_weights(I.TINY, 1)
    S, total = len(blocks), rows * len(blocks)
    rng = np.random.default_rng(rows + sum(blocks))
    toks = torch.from_numpy(rng.integers(0, I.TINY.vocab, total).astype(np.int32)).cuda()
    cu = torch.arange(0, total + 1, rows, dtype=torch.int32, device="cuda")
    lens = [64 * b - rows if 64 * b > rows else 1 for b in blocks]       # the call's last row is its last block's last key
    outs, v_max = [], 0.0
    for flags in (0, B.HSD_FLAG_DETERMINISTIC):
        model = R.DeviceModel(I.TINY, weights, flags)
        kv = R.KvCache(model, [n + rows for n in lens])
        g = torch.Generator(device="cuda").manual_seed(7)
        kv.k_pool.copy_(torch.randn(kv.k_pool.shape, generator=g, device="cuda") * 2)
        kv.v_pool.copy_(torch.randn(kv.v_pool.shape, generator=g, device="cuda"))
        kv.seq_lens.copy_(torch.tensor(lens, dtype=torch.int32))
        eng = R.Engine(model, kv, total, S)
        out = torch.empty(total, I.TINY.n_heads * I.TINY.head_dim, dtype=torch.bfloat16, device="cuda")
        B.check(B.hsd_debug_tap(model.ctx, 0, B.HSD_TAP_ATTN, out, 2 * out.numel()))
        eng.verify_regions(toks, cu, rows, total)
        torch.cuda.synchronize()
        outs.append(out.float().cpu().numpy())
        v_max = max(v_max, float(kv.v_pool[0].float().abs().max()))
    # Either is a mean of V rows with weights rounded to bf16 (2^-9 of the mean of |V|) and is rounded to bf16 (2^-9)
    assert np.abs(outs[0] - outs[1]).max() <= 4 * 2.0 ** -9 * v_max
