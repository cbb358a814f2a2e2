"""Calls with more sequences than rows (most sequences have none): every per-row and per-sequence result of the sequences
that have rows equals that of a call without the empty ones, on a context whose results do not depend on the batch."""
import numpy as np
import pytest

from paper_2602_12957_b200 import inputs as I

pytestmark = pytest.mark.gpu

HAVE = {0: 3, 7: 1, 500: 4, 699: 2}                  # sequence -> rows (10 in all)


def _engine(S):
    import torch
    from paper_2602_12957_b200 import binding as B
    from paper_2602_12957_b200 import runtime as R
    model = R.DeviceModel(I.TINY, I.make_weights(I.TINY, 1), B.HSD_FLAG_DETERMINISTIC)
    kv = R.KvCache(model, [64] * S)
    g = torch.Generator(device="cuda").manual_seed(3)
    kv.k_pool.copy_(torch.randn(kv.k_pool.shape, generator=g, device="cuda"))
    kv.v_pool.copy_(torch.randn(kv.v_pool.shape, generator=g, device="cuda"))
    kv.seq_lens.fill_(20)
    eng = R.Engine(model, kv, sum(HAVE.values()), S)
    eng.ws._raw.fill_(0x55)                           # nothing an unset word happens to be right with
    return eng


@pytest.mark.parametrize("prefill", [False, True])
@pytest.mark.parametrize("S", [700, 1500])
def test_more_sequences_than_rows(S, prefill):
    import torch
    eng = _engine(S)
    rows = np.array([HAVE.get(i, 0) for i in range(S)])
    some = sorted(HAVE)
    toks = eng._i32(np.random.default_rng(2).integers(0, I.TINY.vocab, rows.sum()))
    got = []
    for seqs in (list(range(S)), some):
        cu = eng._i32(np.concatenate([[0], np.cumsum(rows[seqs])]))
        slots, total, longest = eng._i32(seqs), int(rows.sum()), max(HAVE.values())
        if prefill:
            from paper_2602_12957_b200 import binding as B
            eng.kv.seq_lens.zero_()
            first = torch.full((len(seqs),), -7, dtype=torch.int32, device="cuda")
            B.check(B.hsd_prefill(eng.model.ctx, eng.kv.c, len(seqs), cu, None, toks, slots, total, longest, first, eng.ws.ptr,
                                  eng.ws.bytes, torch.cuda.current_stream().cuda_stream))
            eng.check_device()
            assert eng.kv.seq_lens.cpu().tolist() == rows.tolist()
            got.append({"first": first.cpu().numpy()})
        else:
            out = eng.verify_regions(toks, cu, longest, total, slots=slots)
            eng.check_device()
            got.append({k: v.cpu().numpy() for k, v in out.items()})
    every, few = got
    if prefill:
        assert np.array_equal(every["first"][some], few["first"])
        return
    assert np.array_equal(every["accept_len"][some], few["accept_len"]) and np.array_equal(every["n_emit"][some], few["n_emit"])
    assert every["accept_len"].sum() == few["accept_len"].sum() and every["n_emit"].sum() == few["n_emit"].sum()
    for i, j in zip(some, range(len(some))):
        n = few["n_emit"][j]
        assert np.array_equal(every["emit_tokens"][i, :n], few["emit_tokens"][j, :n])
    for k in ("row_argmax", "row_zmax", "row_zdraft"):
        assert np.array_equal(every[k], few[k], equal_nan=k == "row_zdraft"), k
    last = np.cumsum(rows[some]) - 1
    assert np.array_equal(np.flatnonzero(np.isnan(every["row_zdraft"])), last)     # every other row has its draft's logit
