"""The GEMM operator at the row counts where its activation box changes (16, 32, 64, 128 rows), with an odd number of
64-column K sub-tiles (the 64-wide tile stages two at a time; the last half stage lies beyond K), and the SwiGLU epilogue of
the 64-wide tile, against a float64 product of the same bf16 inputs."""
import numpy as np
import pytest

from paper_2602_12957_b200 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def model():
    from paper_2602_12957_b200 import runtime as R
    return R.DeviceModel(I.TINY, I.make_weights(I.TINY, 1))


@pytest.mark.parametrize("tile", [0, 64, 128])
@pytest.mark.parametrize("M", [1, 15, 16, 17, 32, 33, 63, 64, 65, 127, 128, 129])
def test_row_edges(model, M, tile):
    import torch
    from paper_2602_12957_b200 import binding as B
    dev, st = model.device, torch.cuda.current_stream().cuda_stream
    try:
        for N, K in ((256, 192), (128, 64), (1024, 1024)):
            rng = np.random.default_rng(M * 7 + N + K)
            A = I.bf16_round(rng.standard_normal((M, K), dtype=np.float32))
            W = I.bf16_round(rng.standard_normal((N, K), dtype=np.float32) * 0.05)
            ref = A.astype(np.float64) @ W.astype(np.float64).T
            tA, tW = (torch.from_numpy(t).to(dev, torch.bfloat16) for t in (A, W))
            for mode in (0, 1, 2):
                want, cols = ref, N
                if mode == 2:
                    cols, g, u = N // 2, ref[:, :N // 2], ref[:, N // 2:]
                    want = g / (1.0 + np.exp(-g)) * u
                # rows behind the M of the call: must stay as they were
                C = torch.full((M + 8, cols), 3.0, dtype=torch.float32 if mode == 1 else torch.bfloat16, device=dev)
                B.check(B.hsd_debug_set_gemm_tile(model.ctx, tile, 0))
                B.check(B.hsd_op_linear(model.ctx, tA, tW, C, M, N, K, mode, st))
                got = C.float().cpu().numpy().astype(np.float64)
                assert np.all(got[M:] == 3.0), (M, N, K, mode)
                got = got[:M] - (3.0 if mode == 1 else 0.0)
                # fp32: 2^-24 per addition of K terms and of the 3.0 it lands on; bf16: one rounding of the result
                tol = (K * 2.0 ** -24 * 8 + 2.0 ** -22 * 4 if mode == 1 else 2.0 ** -8) * max(1.0, np.abs(want).max()) + 1e-6
                assert np.abs(got - want).max() <= tol, (M, N, K, mode, np.abs(got - want).max(), tol)
    finally:
        B.hsd_debug_set_gemm_tile(model.ctx, 0, 0)
