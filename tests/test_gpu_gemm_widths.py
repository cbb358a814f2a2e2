"""The GEMM operator on tiles whose width does not divide the number of output columns (96, 160, 192, 224: the last tile reaches
beyond the weight's last row and the output's last column) and on pairs of CTAs of every width, with row counts around the
tile's 128 and 256 and K slices of unequal length, against a float64 product of the same bf16 inputs."""
import numpy as np
import pytest

from paper_2602_12957_b200 import inputs as I

pytestmark = pytest.mark.gpu

WIDTHS = [64, 96, 128, 160, 192, 224, 256] + [256 + n for n in (96, 128, 160, 192, 224, 256)]
HAS = {0: (64, 128, 192, 256, 384, 448, 512), 1: tuple(n for n in WIDTHS if n != 224),
       2: tuple(n for n in WIDTHS if n not in (96, 352))}


@pytest.fixture(scope="module")
def model():
    from paper_2602_12957_b200 import runtime as R
    return R.DeviceModel(I.TINY, I.make_weights(I.TINY, 1))


@pytest.mark.parametrize("tile", WIDTHS)
@pytest.mark.parametrize("M,N,K", [(1, 512, 192), (127, 1024, 320), (129, 512, 64), (257, 1280, 448), (1323, 1024, 1024)])
def test_widths(model, tile, M, N, K):
    import torch
    from paper_2602_12957_b200 import binding as B
    dev, st = model.device, torch.cuda.current_stream().cuda_stream
    rng = np.random.default_rng(M + N + K)
    A = I.bf16_round(np.abs(rng.standard_normal((M, K), dtype=np.float32)) + 0.1)      # positive: an output left out is wrong
    W = I.bf16_round(np.abs(rng.standard_normal((N, K), dtype=np.float32)) * 0.05 + 0.01)
    tA, tW = (torch.from_numpy(t).to(dev, torch.bfloat16) for t in (A, W))
    ref = A.astype(np.float64) @ W.astype(np.float64).T
    try:
        for mode in (m for m in (0, 1, 2) if tile in HAS[m]):
            want = ref
            if mode == 2:
                g, u = ref[:, :N // 2], ref[:, N // 2:]
                want = g / (1.0 + np.exp(-g)) * u
            for slices in ((1, 2, 3, 4) if mode == 1 and K > 320 else (0,)):
                # rows behind the output: must stay as they were (a store beyond the last column of a row lands in the next one,
                # that of the last row in these)
                C = torch.full((M + 8, want.shape[1]), 3.0, dtype=torch.float32 if mode == 1 else torch.bfloat16, device=dev)
                B.check(B.hsd_debug_set_gemm_tile(model.ctx, tile, slices))
                B.check(B.hsd_op_linear(model.ctx, tA, tW, C, M, N, K, mode, st))
                got = C.float().cpu().numpy().astype(np.float64)
                assert np.all(got[M:] == 3.0)
                got = got[:M] - (3.0 if mode == 1 else 0.0)
                # fp32: 2^-24 per addition of K terms and of the 3.0 it lands on; bf16: one rounding of the result
                tol = (K * 2.0 ** -24 * 8 + 2.0 ** -22 * 4 if mode == 1 else 2.0 ** -8) * max(1.0, np.abs(want).max()) + 1e-6
                assert np.abs(got - want).max() <= tol, (mode, slices, np.abs(got - want).max(), tol)
    finally:
        B.hsd_debug_set_gemm_tile(model.ctx, 0, 0)


# tile, mode, rows: widths that a mode does not have, and those that only its pairs have (whose place one CTA takes up to 64 rows)
@pytest.mark.parametrize("tile,mode,M,allowed", [
    (224, 0, 129, False), (224, 1, 129, False), (224, 1, 16, False), (224, 2, 129, True), (480, 0, 64, False), (480, 0, 129, False),
    (480, 1, 64, True), (480, 1, 129, True), (480, 2, 64, True), (320, 0, 64, False), (320, 1, 64, False), (320, 1, 129, False),
    (96, 0, 64, False), (96, 1, 64, True), (352, 0, 64, False), (100, 1, 64, False)])
def test_forced_widths_are_taken_or_refused(model, tile, mode, M, allowed):
    import torch
    from paper_2602_12957_b200 import binding as B
    N, K = 512, 128
    A, W = (torch.ones(n, K, dtype=torch.bfloat16, device=model.device) for n in (M, N))
    C = torch.zeros(M, N // 2 if mode == 2 else N, dtype=torch.float32 if mode == 1 else torch.bfloat16, device=model.device)
    try:
        B.check(B.hsd_debug_set_gemm_tile(model.ctx, tile, 0))
        st = B.hsd_op_linear(model.ctx, A, W, C, M, N, K, mode, torch.cuda.current_stream().cuda_stream)
    finally:
        B.hsd_debug_set_gemm_tile(model.ctx, 0, 0)
    assert st == (B.HSD_OK if allowed else B.HSD_ERR_CUDA)
    # refused: nothing was launched; sums of K ones are exact (SwiGLU of 128: 128 * 128)
    assert bool((C == ((K * K if mode == 2 else K) if allowed else 0)).all())
