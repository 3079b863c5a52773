"""The BF16 loss and gradient of as many pairs as a call takes: 65,536 tiles of 32
stacked rows, one more than a grid's second dimension."""
import numpy as np
import pytest

F = pytest.importorskip("paper_2606_15476_gb300.farm")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1048544, 1048550, 1 << 20])
def test_last_pairs_count(n):
    dim, h, p, few = 4, 64, 64, 40
    rng = np.random.default_rng(n)
    f = lambda *s: rng.standard_normal(s).astype(np.float32)  # noqa: E731
    xq, xd, y = f(n, dim), f(n, dim), rng.uniform(-1, 1, n).astype(np.float32)
    w = np.zeros(n, np.float32)
    w[-few:] = 1.0
    ctx = F.farm_create(0)
    try:
        F.farm_mlp_set(ctx, f(h, dim) / 2, f(h) / 4, f(p, h) / 8, f(p) / 4)
        count = h * dim + h + p * h + p
        loss, grad = F.farm_mlp_loss_grad(ctx, xq, xd, y, w, count, F.PREC_BF16)
        loss1, grad1 = F.farm_mlp_loss_grad(ctx, xq[-few:], xd[-few:], y[-few:], w[-few:], count, F.PREC_BF16)
    finally:
        F.farm_destroy(ctx)
    # the other pairs' terms are exactly zero: sums of the same 80 terms in another
    # order, each within 80 x 2^-23 of the sum of their magnitudes
    assert abs(loss - loss1) <= 1e-5 * abs(loss1)
    np.testing.assert_allclose(grad, grad1, rtol=0, atol=1e-5 * np.abs(grad1).max())
    assert np.abs(grad1).max() > 0
