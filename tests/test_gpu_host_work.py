"""The host's work around a call's launches does not grow with the decoder's depth: GEMM tiles are chosen when a context is
created, for calls of up to 8,192 rows, and once per projection of a larger call.  A context's creation loads the kernels and encodes the maps of the tile widths that its
projections can be given, and no others."""
import numpy as np
import pytest

from paper_2602_12957_b200 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layers", [1, 7])
def test_tile_choices(layers):
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

    assert choices(lambda: eng.prefill([None, None], [np.arange(13), np.arange(7)])) == 0
    assert choices(lambda: eng.verify_regions(toks, cu, 13, 20)) == 0
    assert choices(lambda: eng.verify_tree(toks, cu, parent, 13, 20)) == 0
    x = torch.zeros(64, 64, dtype=torch.bfloat16, device=model.device)
    st = torch.cuda.current_stream().cuda_stream
    assert choices(lambda: B.check(B.hsd_op_linear(model.ctx, x, x, x.clone(), 64, 64, 64, 0, st))) == 1
    for rows, n in ((8192, 0), (8193, 4)):                # (the LM head of a prefill has a row a sequence)
        kv = R.KvCache(model, [rows])
        eng = R.Engine(model, kv, rows, 1)
        assert choices(lambda: eng.prefill([None], [np.arange(rows) % cfg.vocab])) == n


# widths of a projection's tiles, pairs' among them: heads of 64 keep whole heads, heads of 128 too; kernels: three for a width of 64
# (at most 16, at most 64 and more rows), and one more for each width that pairs have too
@pytest.mark.parametrize("head_dim,qkv_maps,qkv_kernels", [(64, 4, 6 + 3), (128, 2, 2 + 2)])
def test_a_context_prepares_its_models_widths_only(head_dim, qkv_maps, qkv_kernels):
    from paper_2602_12957_b200 import binding as B
    from paper_2602_12957_b200 import runtime as R
    cfg = I.ModelConfig(n_layers=3, d_model=512, n_heads=4, n_kv_heads=2, head_dim=head_dim, d_ffn=1024, vocab=1024)
    model = R.DeviceModel(cfg, I.make_weights(cfg, 1))
    for m in (model, model.sibling(B.HSD_FLAG_DETERMINISTIC)):
        work = B.hsd_debug_host_work(m.ctx)[1]
        # residual adds 64, 96 .. 256, SwiGLU the same without 96, LM head 64, 128, 256
        assert work["weight_maps"] == 3 * (qkv_maps + 7 + 6 + 7) + 3
        assert work["gemm_kernels"] == qkv_kernels + (8 + 6) + (8 + 5) + (5 + 2)
        assert work["tile_choices"] == 5 * (3 + 64)
