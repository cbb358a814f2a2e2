"""The workspace of small calls: what the partial results of cut KV ranges take is bounded by the call's own q-tiles, a
larger call never needs less, and a long context is worked inside exactly the bytes that were asked for."""
import numpy as np
import pytest

from paper_2602_12957_b200 import inputs as I
from . import harness as H

pytestmark = pytest.mark.gpu

CFGS = {"hd64": I.ModelConfig(n_layers=1, d_model=1024, n_heads=16, n_kv_heads=8, head_dim=64, d_ffn=1024, vocab=4096),
        "hd128": I.ModelConfig(n_layers=1, d_model=2048, n_heads=16, n_kv_heads=8, head_dim=128, d_ffn=1024, vocab=4096,
                               qk_norm=True)}


@pytest.fixture(scope="module", params=list(CFGS))
def model(request):
    from paper_2602_12957_b200 import runtime as R
    return R.DeviceModel(CFGS[request.param], I.make_weights(CFGS[request.param], 1))


def test_sizes(model):
    from paper_2602_12957_b200 import binding as B
    size = lambda T, S: B.hsd_workspace_bytes(model.ctx, T, S)  # noqa: E731
    eight = 8 * model.cfg.n_kv_heads * 128 * (model.cfg.head_dim + 2) * 4    # bytes of eight slices of a q-tile
    assert size(1, 1) < eight + (1 << 17)
    assert size(64, 1) < 2 * eight + (3 << 20)
    rows = list(range(1, 200)) + [512, 513, 2049, 9000]
    for S in (1, 2, 3, 7, 16, 66):
        sizes = [size(T, S) for T in rows]
        assert all(a <= b for a, b in zip(sizes, sizes[1:])), S
        assert all(size(T, S) <= size(T, S + 1) for T in rows)


@pytest.mark.parametrize("rows,blocks", [(1, [200]), (17, [200]), (48, [200]), (63, [150]), (64, [150]), (20, [90, 60, 5])])
def test_long_context_in_the_bytes_asked_for(model, rows, blocks):
    import torch
    from paper_2602_12957_b200 import runtime as R
    cfg, n, guard = model.cfg, len(blocks), 1 << 16
    lens, per = [64 * b - rows for b in blocks], [rows] * n
    kv = R.KvCache(model, [64 * b for b in blocks])
    g = torch.Generator(device="cuda").manual_seed(7)
    kv.k_pool.copy_(torch.randn(kv.k_pool.shape, generator=g, device="cuda") * 3)
    kv.v_pool.copy_(torch.randn(kv.v_pool.shape, generator=g, device="cuda"))
    eng = R.Engine(model, kv, rows * n, n)
    held = torch.full((eng.ws.bytes + 1024 + guard,), 0x55, dtype=torch.uint8, device="cuda")
    off = (-held.data_ptr()) % 1024
    eng.ws._raw, eng.ws.ptr = held, held.data_ptr() + off
    toks = eng._i32(np.random.default_rng(rows).integers(0, cfg.vocab, rows * n))
    q, out = H.layer0_attention(eng, toks, eng._i32(np.arange(n + 1) * rows), lens, per)
    assert bool((held[off + eng.ws.bytes:] == 0x55).all()) and bool((held[:off] == 0x55).all())
    want, spread = H.attention_float64(cfg, kv, q, lens, per)
    over = (out.double() - want).abs() - H.attention_tolerance(want, spread)
    assert float(over.max()) <= 0
