"""The association on both sides of the size from which it keeps only the
cosines reaching tau_f: a large call against calls of 100 detections, which
store their rows (a detection's matches depend on it and the entities alone),
with lists longer than the 2,048 entries of a buffer among them."""
import numpy as np
import pytest

from test_gpu_assoc_lists import F, _world

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,b,n_cls", [(8987, 700, 3), (8988, 700, 3), (49000, 129, 20), (3000, 2100, 40)])
def test_matches_equal_those_of_small_calls(n, b, n_cls):
    ent, det = _world(np.random.default_rng(n), n, b, 64, n_cls, 20.0)
    ctx = F.farm_create(0)
    try:
        whole = F.farm_associate(ctx, ent, det, 0.8, 0.9, 8)
        for d0 in range(0, b, 100):
            part = {k: np.ascontiguousarray(v[d0:d0 + 100] if k == "feat" else v[:, d0:d0 + 100]) for k, v in det.items()}
            got = F.farm_associate(ctx, ent, part, 0.8, 0.9, 8)
            for k in ("match_cnt", "match_idx", "match_h"):
                np.testing.assert_array_equal(whole[k][d0:d0 + 100], got[k])
    finally:
        F.farm_destroy(ctx)
