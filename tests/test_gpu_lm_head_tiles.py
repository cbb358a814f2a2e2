"""The LM head of calls with one tile of rows waits for its weights and is slower on 256-wide tiles: the tiles of calls of 1 to 128
rows are narrower (or pairs'), whatever the vocabulary and K, and the argmax is that of a float64 product."""
import pytest

from paper_2602_12957_b200 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("vocab,d", [(32768, 2048), (65536, 512), (131072, 256)])
@pytest.mark.parametrize("rows", [1, 16, 17, 32, 64, 65, 128])
def test_one_row_tile(vocab, d, rows):
    import torch
    from paper_2602_12957_b200 import binding as B
    cfg = I.ModelConfig(n_layers=1, d_model=d, n_heads=2, n_kv_heads=2, head_dim=64, d_ffn=128, vocab=vocab)
    gen = torch.Generator("cuda").manual_seed(rows + d)
    new = lambda *shape: torch.randn(*shape, device="cuda", generator=gen).to(torch.bfloat16)  # noqa: E731
    lm, one = new(vocab, d), [new(max(2 * 128, 6 * 64) * d)]        # (the layer's weights are not read here)
    st, ctx = B.hsd_create(B.make_config(cfg), B.make_weights(lm, lm, one[0], one, one, one, one, one, one))
    B.check(st)
    h = new(rows, d)
    best, am = torch.empty(rows, dtype=torch.int64, device="cuda"), torch.empty(rows, dtype=torch.int32, device="cuda")
    zmax = torch.empty(rows, device="cuda")
    try:
        B.check(B.hsd_op_lm_head_argmax(ctx, h, rows, None, best, rows * 8, am, zmax, None, torch.cuda.current_stream().cuda_stream))
        torch.cuda.synchronize()
        st, (columns, _, pair) = B.hsd_debug_tile(ctx, 4, rows)
    finally:
        B.hsd_destroy(ctx)
    assert st == B.HSD_OK and (columns < 256 or pair), (columns, pair)
    z = h.double() @ lm.double().T
    top = z.max(1).values
    # fp32 sums of d products: 2^-24 an addition, of terms that the rows' norms bound
    tol = 2.0 ** -24 * d ** 0.5 * 8 * float(h.double().norm(dim=1).max() * lm.double().norm(dim=1).max())
    assert float((zmax.double() - top).abs().max()) <= tol
    assert float((top - z.gather(1, am.long()[:, None])[:, 0]).max()) <= 2 * tol
