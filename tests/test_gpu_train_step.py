"""The tensor-core training step at the edges of its tiles (32 rows x 64
columns, 32 pairs per block, contractions padded to 64 rows), against the FP32
CUDA-core forward and backward.  Bounds: each operand of the contractions is
rounded to BF16 (relative error 2^-9), twice per product and through four
contractions in a row, which stays below 3e-2 of the gradient's norm; the loss
below 1e-2."""
import numpy as np
import pytest

F = pytest.importorskip("paper_2606_15476_gb300.farm")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pairs", [1, 31, 33, 65, 300])
@pytest.mark.parametrize("D,H,P", [(72, 64, 64), (130, 192, 128), (64, 128, 320), (200, 64, 1024)])
def test_gradient_against_fp32(pairs, D, H, P):
    rng = np.random.default_rng(pairs + D)
    ws = [rng.standard_normal((H, D)) / np.sqrt(D), 0.1 * rng.standard_normal(H),
          rng.standard_normal((P, H)) / np.sqrt(H), 0.1 * rng.standard_normal(P)]
    xq, xd = (rng.standard_normal((pairs, D)) for _ in range(2))
    xq, xd = (x / np.linalg.norm(x, axis=1, keepdims=True) for x in (xq, xd))
    y = rng.uniform(-1.0, -0.5, pairs)          # far from the cosines: no residual cancels
    w = rng.integers(1, 5, pairs)
    n = H * D + H + P * H + P
    ctx = F.farm_create(0)
    try:
        F.farm_mlp_set(ctx, *ws)
        for wt in (None, w):
            l16, g16 = F.farm_mlp_loss_grad(ctx, xq, xd, y, wt, n, F.PREC_BF16)
            l32, g32 = F.farm_mlp_loss_grad(ctx, xq, xd, y, wt, n, F.PREC_FP32_SIMT)
            assert abs(l16 - l32) <= 1e-2 * l32
            at = np.cumsum([0, H * D, H, P * H, P])
            for a, b in zip(at[:-1], at[1:]):
                assert np.linalg.norm(g16[a:b] - g32[a:b]) <= 3e-2 * np.linalg.norm(g32[a:b])
    finally:
        F.farm_destroy(ctx)
