"""The host's work around a call's launches does not grow with the decoder's depth: GEMM tiles are chosen once per projection
of a call and once for its LM head."""
import numpy as np
import pytest

from paper_2602_12957_b200 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layers", [1, 7])
def test_one_tile_choice_per_projection_and_call(layers):
    import torch
    from paper_2602_12957_b200 import binding as B
    from paper_2602_12957_b200 import runtime as R
    cfg = I.ModelConfig(n_layers=layers, d_model=256, n_heads=4, n_kv_heads=2, head_dim=64, d_ffn=512, vocab=1024)
    model = R.DeviceModel(cfg, I.make_weights(cfg, 1))
    kv = R.KvCache(model, [128, 128])
    eng = R.Engine(model, kv, 40, 2)
    toks, cu = eng._i32(np.arange(20)), eng._i32([0, 13, 20])
    parent = eng._i32([-1] + list(range(12)) + [-1] + list(range(6)))

    def choices(call):
        before = B.hsd_debug_host_work(model.ctx)[1]["tile_choices"]
        call()
        eng.check_device()
        return B.hsd_debug_host_work(model.ctx)[1]["tile_choices"] - before

    assert choices(lambda: eng.prefill([None, None], [np.arange(13), np.arange(7)])) == 5
    assert choices(lambda: eng.verify_regions(toks, cu, 13, 20)) == 5
    assert choices(lambda: eng.verify_tree(toks, cu, parent, 13, 20)) == 5
    x = torch.zeros(64, 64, dtype=torch.bfloat16, device=model.device)
    st = torch.cuda.current_stream().cuda_stream
    assert choices(lambda: B.check(B.hsd_op_linear(model.ctx, x, x, x.clone(), 64, 64, 64, 0, st))) == 1
