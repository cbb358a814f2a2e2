"""The host-buffer call at input and result areas of every remainder mod 4 words (they travel 16 bytes at a time): the
integers of the device call on the same inputs, exactly, and nothing written outside the result buffers."""
import numpy as np
import pytest

from paper_2602_12957_b200 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [[1], [2], [3], [1, 1], [1, 4], [5, 2, 9], [1, 1, 1, 1], [17, 1, 33], [128, 1, 3, 64, 7]])
def test_ragged_areas(rows):
    import torch
    from paper_2602_12957_b200 import binding as B
    from paper_2602_12957_b200 import runtime as R
    model = R.DeviceModel(I.TINY, I.make_weights(I.TINY, 1), B.HSD_FLAG_DETERMINISTIC)
    kv = R.KvCache(model, [n + 1 for n in rows])
    S, total, longest = len(rows), sum(rows), max(rows)
    eng = R.Engine(model, kv, total, S)
    rng = np.random.default_rng(total)
    toks = rng.integers(0, I.TINY.vocab, total).astype(np.int32)
    cu = np.concatenate([[0], np.cumsum(rows)]).astype(np.int32)
    out = eng.verify_regions(torch.from_numpy(toks).cuda(), torch.from_numpy(cu).cuda(), longest, total)
    want = {k: out[k].cpu().numpy() for k in ("accept_len", "n_emit", "emit_tokens")}
    acc, nem, emit = (np.full(n + 8, -7, np.int32) for n in (S, S, S * longest))
    rc, mq = B.hsd_verify_regions_host(model.ctx, kv.c, S, torch.from_numpy(cu), torch.from_numpy(toks), None, 0.0, 1,
                                       *(torch.from_numpy(a) for a in (acc, emit, nem)), eng.ws.ptr, eng.ws.bytes,
                                       torch.cuda.current_stream().cuda_stream)
    B.check(rc, "hsd_verify_regions_host")
    assert mq == longest
    assert acc[:S].tolist() == want["accept_len"].tolist() and nem[:S].tolist() == want["n_emit"].tolist()
    for i in range(S):
        n = int(nem[i])
        assert emit[i * longest:i * longest + n].tolist() == want["emit_tokens"].reshape(S, -1)[i, :n].tolist()
    for a in (acc[S:], nem[S:], emit[S * longest:]):
        assert (a == -7).all()
    assert kv.seq_lens.cpu().numpy().tolist() == nem[:S].tolist()
