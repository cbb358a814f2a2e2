"""A tree node's own logit under its parent's distribution, at the model widths whose rows a warp holds in 1 to 32 pieces: against
the plain kernel's logits of the normed rows, with the argmax's logit taken over bit by bit where the node carries it, and NaN
for roots and padding rows."""
import numpy as np
import pytest

from paper_2602_12957_b200 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [128, 256, 512, 1024, 2048, 4096])
@pytest.mark.parametrize("rows", [[1], [9, 1, 128]])
def test_child_logits(d, rows):
    import torch
    from paper_2602_12957_b200 import binding as B
    from paper_2602_12957_b200 import runtime as R
    cfg = I.ModelConfig(n_layers=1, d_model=d, n_heads=2, n_kv_heads=2, head_dim=64, d_ffn=128, vocab=4096)
    model = R.DeviceModel(cfg, I.make_weights(cfg, 3))
    S, T = len(rows), sum(rows)
    kv = R.KvCache(model, [n + 64 for n in rows])
    kv.k_pool.zero_()
    kv.v_pool.zero_()
    kv.seq_lens.fill_(20)
    eng = R.Engine(model, kv, 2 * T, S)
    rng = np.random.default_rng(d + T)
    parent = np.concatenate([[-1] + [int(rng.integers(0, j)) for j in range(1, n)] for n in rows]).astype(np.int32)
    cu = np.concatenate([[0], np.cumsum(rows)]).astype(np.int32)
    if rows[-1] == 128:
        parent[-3:] = -2                                                    # padding rows
    toks = rng.integers(0, cfg.vocab, T).astype(np.int32)
    out = eng.verify_tree(eng._i32(toks), eng._i32(cu), eng._i32(parent), max(rows), T, log_tau=-0.3)
    # a second call in which some nodes carry their parent's argmax (a node's row depends on its ancestors' tokens only, so a
    # leaf can be changed without changing its parent)
    am = out["row_argmax"].cpu().numpy()
    base = np.repeat(cu[:-1], rows)
    leaf = [r for r in range(T) if parent[r] >= 0 and not ((parent + base == r) & (parent >= 0)).any()]
    hit = leaf[::3]
    for r in hit:
        toks[r] = am[base[r] + parent[r]]
    out = eng.verify_tree(eng._i32(toks), eng._i32(cu), eng._i32(parent), max(rows), T, log_tau=-0.3)
    logits = torch.empty(2 * T, cfg.vocab, device="cuda")
    B.check(B.hsd_debug_logits(model.ctx, eng.ws.ptr, 2 * T, S, logits, torch.cuda.current_stream().cuda_stream))
    z, zmax = out["row_zchild"].cpu().numpy(), out["row_zmax"].cpu().numpy()
    # sums of d products in fp32 in different orders: 2^-24 per addition, of terms bounded by the row's norm times the weight's
    scale = float(model.lm_head.float().norm(dim=1).max()) * np.sqrt(d)
    for r in range(T):
        if parent[r] < 0:
            assert np.isnan(z[r]), r
            continue
        p = base[r] + parent[r]
        assert abs(z[r] - float(logits[p, int(toks[r])])) <= 2.0 ** -24 * np.sqrt(d) * 8 * scale, (r, z[r])
    am = out["row_argmax"].cpu().numpy()
    same = [r for r in hit if toks[r] == am[base[r] + parent[r]]]
    assert all(z[r] == zmax[base[r] + parent[r]] for r in same) and (len(same) > 0 or not hit)
