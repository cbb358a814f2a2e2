"""Counts beyond what a kernel takes at once: more drafts per sequence than are searched together (64), accepted paths of more
depths than are moved together (16), more sequences than a set-up CTA keeps the offsets of (1,024) and more q-tiles than the
attention plan keeps the lengths of (512)."""
import numpy as np
import pytest

from paper_2602_12957_b200 import inputs as I
from . import harness as H
from .test_gpu_dsv import _engine, check_build

pytestmark = pytest.mark.gpu


def test_more_drafts_than_are_searched_together():
    eng, _, _ = _engine()
    rng = np.random.default_rng(23)
    for n_drafts in (63, 64, 65, 128, 129, 200):
        for n, vocab, longest in ((1, 40, 30), (3, 3, 12), (8, 2, 20), (2, 30, 90)):
            S = 3
            windows = [rng.integers(0, vocab, size=n).tolist() for _ in range(S)]
            # empty drafts and drafts no longer than the window among them; sequences of other counts beside
            drafts = [[rng.integers(0, vocab, size=int(rng.integers(0, longest))).tolist() for _ in range(k)]
                      for k in (n_drafts, 0, n_drafts // 2)]
            check_build(eng, windows, drafts, int(rng.choice([128, 33, 2])))


@pytest.mark.parametrize("head_dim", [64, 128])
def test_long_accepted_paths(head_dim):
    import torch
    from paper_2602_12957_b200 import runtime as R
    cfg = I.ModelConfig(n_layers=2, d_model=256, n_heads=4, n_kv_heads=2, head_dim=head_dim, d_ffn=256, vocab=256)
    model = R.DeviceModel(cfg, I.make_weights(cfg, 1))
    rng = np.random.default_rng(head_dim)
    depths = [127, 0, 1, 15, 16, 17, 33, 64, 100, -1]
    lens = [0, 5, 63, 64, 1, 127, 60, 30, 129, 7]
    S, rows = len(depths), 128
    kv = R.KvCache(model, [n + rows for n in lens])
    g = torch.Generator(device="cuda").manual_seed(3)
    for pool in (kv.k_pool, kv.v_pool):
        pool.copy_(torch.randn(pool.shape, generator=g, device="cuda"))
    kv.seq_lens.copy_(torch.tensor(lens, dtype=torch.int32))
    path = np.full((S, rows), -5, np.int32)
    for i, a in enumerate(depths):
        if a > 0:
            path[i, :a] = np.sort(rng.choice(np.arange(1, rows), size=a, replace=False))      # any increasing rows
    want = [p.cpu().view(torch.int16).numpy().copy() for p in (kv.k_pool, kv.v_pool)]
    for pool in want:
        old = pool.copy()
        for i, a in enumerate(depths):
            for d in range(1, a + 1):
                src, dst = lens[i] + path[i, d - 1], lens[i] + d
                pool[:, kv.table_host[i, dst // 64], :, dst % 64] = old[:, kv.table_host[i, src // 64], :, src % 64]
    eng = R.Engine(model, kv, rows, S)
    eng.commit_tree(eng._i32(depths), eng._i32(path.reshape(-1)).reshape(S, rows))
    torch.cuda.synchronize()
    for pool, w in zip((kv.k_pool, kv.v_pool), want):
        assert np.array_equal(pool.cpu().view(torch.int16).numpy(), w)
    assert kv.seq_lens.cpu().tolist() == [n + a + 1 for n, a in zip(lens, depths)]


def test_more_sequences_and_tiles_than_are_kept():
    from paper_2602_12957_b200 import runtime as R
    import torch
    cfg, S = I.TINY, 1500
    model = R.DeviceModel(cfg, I.make_weights(cfg, 1))
    rng = np.random.default_rng(9)
    rows = rng.integers(1, 4, S).tolist()
    lens = rng.integers(0, 190, S).tolist()
    lens[1200] = 1800                                     # (one long range among them)
    kv = R.KvCache(model, [a + b for a, b in zip(lens, rows)])
    g = torch.Generator(device="cuda").manual_seed(7)
    kv.k_pool.copy_(torch.randn(kv.k_pool.shape, generator=g, device="cuda") * 8)
    kv.v_pool.copy_(torch.randn(kv.v_pool.shape, generator=g, device="cuda"))
    eng = R.Engine(model, kv, sum(rows), S)
    toks = eng._i32(rng.integers(0, cfg.vocab, sum(rows)))
    q, out = H.layer0_attention(eng, toks, eng._i32(np.concatenate([[0], np.cumsum(rows)])), lens, rows)
    want, spread = H.attention_float64(cfg, kv, q, lens, rows)
    assert float(((out.double() - want).abs() / H.attention_tolerance(want, spread)).max()) <= 1
