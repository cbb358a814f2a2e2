"""Ties and near-ties between a tree node's children.  A child's logit is summed in another order than its parent's maximum, so
a sibling whose LM-head row equals the argmax's, or differs from it by one rounding, may come out on either side of it; the
traversal must take the child that carries the argmax all the same, and no child's logit may lie above its parent's maximum."""
import numpy as np
import pytest

from paper_2602_12957_b200 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("near", [False, True])       # the sibling's row equals the argmax's / is one bf16 step off in one column
@pytest.mark.parametrize("d", [256, 1024])
def test_argmax_child_wins(d, near):
    import torch
    from paper_2602_12957_b200 import binding as B
    from paper_2602_12957_b200 import runtime as R
    cfg = I.ModelConfig(n_layers=1, d_model=d, n_heads=2, n_kv_heads=2, head_dim=64, d_ffn=128, vocab=4096)
    model = R.DeviceModel(cfg, I.make_weights(cfg, 5))
    S, n = 64, 3                                          # a root and two children each
    kv = R.KvCache(model, [64] * S)
    eng = R.Engine(model, kv, 2 * S * n, S)
    roots = np.random.default_rng(d).permutation(cfg.vocab)[:S]
    parent, cu = np.tile(np.array([-1, 0, 0], np.int32), S), np.arange(S + 1, dtype=np.int32) * n

    def step(first, second):
        toks = np.stack([roots, first, second], 1).reshape(-1)
        out = eng.verify_tree(eng._i32(toks), eng._i32(cu), eng._i32(parent), n, S * n, log_tau=-0.3)
        eng.check_device("verify_tree")
        return {k: v.cpu().numpy() for k, v in out.items()}

    top = step(roots, roots)["row_argmax"].reshape(S, n)[:, 0]
    # every argmax gets a twin: a token that is no one's argmax, above or below it in turn
    free = np.setdiff1d(np.arange(cfg.vocab), top)
    twin, used = {}, set()
    for k, t in enumerate(sorted(set(top.tolist()))):
        side = free[free > t] if k % 2 and t < cfg.vocab - S else free[free < t] if t > S else free
        twin[t] = next(int(v) for v in side if int(v) not in used)
        used.add(twin[t])
        row = model.lm_head[t].clone()
        if near:
            j = int(row.abs().argmin())                   # the smallest weight: its step moves the logit by less than a rounding
            row[j] = row[j] * (1.0 + 2.0 ** -7)
        model.lm_head[twin[t]] = row
    twins = np.array([twin[int(t)] for t in top])
    for first, second in ((top, twins), (twins, top)):
        out = step(first, second)
        rows = {k: out[k].reshape(S, n) for k in ("row_argmax", "row_zmax", "row_zchild")}
        both = np.stack([first, second], 1)
        hat = rows["row_argmax"][:, 0]
        assert np.all((both == hat[:, None]).sum(1) == 1)                     # one of the two carries it
        if not near:
            assert np.array_equal(hat, both.min(1))                           # equal rows: the lower id
        z, zmax = rows["row_zchild"][:, 1:], rows["row_zmax"][:, 0]
        # the sums run over d products in two orders: 2^-24 an addition, of terms that the row norms bound
        scale = float(model.lm_head.float().norm(dim=1).max()) * np.sqrt(d)
        assert np.all(zmax[:, None] - z <= 2.0 ** -24 * np.sqrt(d) * 8 * scale + (2.0 ** -7 * scale / d if near else 0.0))
        assert np.all(z <= zmax[:, None]), (z - zmax[:, None]).max()
        won = both[np.arange(S), out["accept_rows"][:, 0] - 1]
        assert np.all(out["accept_len"] >= 1) and np.array_equal(won, hat), np.flatnonzero(won != hat)
