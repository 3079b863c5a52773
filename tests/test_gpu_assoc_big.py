"""The fusion of components with many members (summed a segment of 1,024 at a
time by whole blocks) against FP64 sums over the same components."""
import numpy as np
import pytest

from test_gpu_assoc_lists import F, _world

pytestmark = pytest.mark.gpu


# (members of a component: about b / n; the first world's stay at the warps' 64)
@pytest.mark.parametrize("n,b,feat", [(8, 400, 64), (3, 250, 7), (1, 1024, 513), (1, 1025, 1152), (5, 9000, 40),
                                      (40, 60000, 256)])
def test_big_components(n, b, feat):
    ent, det = _world(np.random.default_rng(b + feat), n, b, feat, n, 40.0)
    ctx = F.farm_create(0)
    try:
        got = F.farm_associate(ctx, ent, det, 0.8, 0.9, 4)
    finally:
        F.farm_destroy(ctx)
    # every component by pointer jumping over the reported matches
    t = n + b
    d, j = np.nonzero(got["match_idx"] >= 0)
    u, v = n + d, got["match_idx"][d, j]
    label = np.arange(t)
    while True:
        low = np.minimum(label[u], label[v])
        new = label.copy()
        np.minimum.at(new, u, low)
        np.minimum.at(new, v, low)
        new = new[new]
        if np.array_equal(new, label):
            break
        label = new
    w = np.concatenate([ent["w"], np.ones(b, np.float32)]).astype(np.float64)
    parent = np.arange(t)
    for c in np.unique(label[:n]):
        es = np.flatnonzero(label[:n] == c)
        parent[label == c] = es[np.lexsort((es, -w[es]))[0]]
    np.testing.assert_array_equal(got["parent"], parent)
    assert np.bincount(parent, minlength=t).max() > min(b, 64) / 2
    mu = np.concatenate([ent["mu"], det["mu"]], axis=1).astype(np.float64)
    cv = np.concatenate([ent["cov"], det["cov"]], axis=1).astype(np.float64)
    ft = np.concatenate([ent["feat"], det["feat"]]).astype(np.float64)

    def total(x):                              # [k, t] summed into the winners
        out = np.zeros((len(x), t))
        for r in range(len(x)):
            out[r] = np.bincount(parent, x[r], t)
        return out
    W = total(w[None])[0]
    own = W > 0
    m = np.divide(total(w * mu), W, out=np.zeros((3, t)), where=own)
    dm = mu - m[:, parent]
    ia, ib = [0, 0, 0, 1, 1, 2], [0, 1, 2, 1, 2, 2]
    c = np.divide(total(w * (cv + dm[ia] * dm[ib])), W, out=np.zeros((6, t)), where=own)
    f = np.divide(total(w * ft.T), W, out=np.zeros((feat, t)), where=own)
    np.testing.assert_array_equal(got["w"], W)
    # FP32: a lane adds at most 128 terms of a segment and 59 segments follow, so sums of
    # terms of one sign are off by at most 2e-5 relative, and the features (at most 1, of
    # either sign) by as much absolutely; coordinates up to 40 are themselves rounded to 2e-6
    np.testing.assert_allclose(got["mu"], m, rtol=0, atol=2e-5)
    np.testing.assert_allclose(got["cov"], c, rtol=1e-4, atol=2e-6)
    np.testing.assert_allclose(got["feat"].T, f, rtol=0, atol=2e-5)
