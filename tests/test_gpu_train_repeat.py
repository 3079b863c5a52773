"""The gradients of the tensor-core training step are summed in one fixed order,
the bias gradients by the last block that reaches their columns: repeated calls
agree bit for bit (2 to 3,000 stacked rows, 256 to a bias sum)."""
import numpy as np
import pytest

F = pytest.importorskip("paper_2606_15476_gb300.farm")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pairs", [1, 128, 129, 400, 1500])
def test_gradients_repeat_bit_for_bit(pairs):
    rng = np.random.default_rng(pairs)
    D, H, P = 72, 128, 320
    ws = [rng.standard_normal((H, D)) / np.sqrt(D), 0.1 * rng.standard_normal(H),
          rng.standard_normal((P, H)) / np.sqrt(H), 0.1 * rng.standard_normal(P)]
    xq, xd = (rng.standard_normal((pairs, D)) for _ in range(2))
    y = rng.uniform(-1.0, -0.5, pairs)
    n = H * D + H + P * H + P
    ctx = F.farm_create(0)
    try:
        F.farm_mlp_set(ctx, *ws)
        g = [F.farm_mlp_loss_grad(ctx, xq, xd, y, None, n, F.PREC_BF16)[1] for _ in range(4)]
        for other in g[1:]:
            np.testing.assert_array_equal(g[0], other)
    finally:
        F.farm_destroy(ctx)
