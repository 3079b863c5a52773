"""The association's search over rows most of whose cosines reach tau_f, so that
its list of entities fills and is emptied pass after pass: match counts against
the Hellinger distances alone, in FP64."""
import numpy as np
import pytest

from test_gpu_assoc_lists import F, _world

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2048, 2049, 6500, 40000])
@pytest.mark.parametrize("tau", [-1.0, 0.0])
def test_dense_rows(n, tau):
    b, feat = 120, 8
    ent, det = _world(np.random.default_rng(n), n, b, feat, 1 if tau == 0.0 else 3, 60.0)
    # (tau 0: one class, whose cosines are all near 1)
    c = lambda x: x.astype(np.float64)  # noqa: E731
    s = 0.5 * (c(ent["cov"])[[0, 3, 5]][:, None, :] + c(det["cov"])[[0, 3, 5]][:, :, None])      # (diagonal covariances)
    d = c(ent["mu"])[:, None, :] - c(det["mu"])[:, :, None]
    ld = lambda x: np.log(c(x["cov"])[[0, 3, 5]]).sum(0)  # noqa: E731
    bc = 0.25 * (ld(ent)[None] + ld(det)[:, None]) - 0.5 * np.log(s).sum(0) - 0.125 * (d * d / s).sum(0)
    h = np.sqrt(np.maximum(-np.expm1(bc), 0.0))
    # (FP32 distances are within 1e-5 of these: lb to ub matches)
    act = ent["active"][None] != 0
    lb, ub = ((h <= 0.9 - 1e-5) & act).sum(1), ((h <= 0.9 + 1e-5) & act).sum(1)
    ctx = F.farm_create(0)
    try:
        for _ in range(10):
            got = F.farm_associate(ctx, ent, det, tau, 0.9, 8)["match_cnt"]
            assert (got >= lb).all() and (got <= ub).all()
    finally:
        F.farm_destroy(ctx)
