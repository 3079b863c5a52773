"""The association's emitted candidate lists (more than 128 detections) against
its stored rows (at most 128), with lists that overflow their buffers, and the
fusion of small, large and lone components against FP64 sums over the same
components."""
import numpy as np
import pytest

F = pytest.importorskip("paper_2606_15476_gb300.farm")
pytestmark = pytest.mark.gpu


def _world(rng, n, b, feat, n_cls, spread):
    cen = rng.standard_normal((n_cls, feat))
    cen /= np.linalg.norm(cen, axis=1, keepdims=True)
    unit = lambda x: (x / np.linalg.norm(x, axis=1, keepdims=True)).astype(np.float32)  # noqa: E731
    cls, src = rng.integers(0, n_cls, n), rng.integers(0, n, b)
    mu = rng.uniform(0, spread, (3, n))
    var = rng.uniform(0.01, 0.1, (3, n))

    def cov(v):
        z = np.zeros(v.shape[1])
        return np.stack([v[0], z, z, v[1], z, v[2]]).astype(np.float32)
    ent = dict(mu=mu.astype(np.float32), cov=cov(var), feat=unit(cen[cls] + 0.01 * rng.standard_normal((n, feat))),
               w=rng.integers(0, 9, n).astype(np.float32), active=(rng.uniform(size=n) > 0.1).astype(np.int32))
    det = dict(mu=(mu[:, src] + 0.05 * rng.standard_normal((3, b))).astype(np.float32), cov=cov(var[:, src]),
               feat=unit(cen[cls[src]] + 0.01 * rng.standard_normal((b, feat))))
    return ent, det


@pytest.mark.parametrize("n,b,feat,n_cls", [(300, 129, 20, 3), (9000, 300, 64, 3), (4097, 200, 256, 2), (70, 400, 7, 40)])
def test_emitted_lists_equal_stored_rows(n, b, feat, n_cls):
    # (9,000 and 4,097 entities of 3 and 2 classes: lists of about 3,000 and
    # 2,050, some above the 2,048 of a buffer)
    rng = np.random.default_rng(n)
    ent, det = _world(rng, n, b, feat, n_cls, 20.0)
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


@pytest.mark.parametrize("n,b,feat,n_cls,spread", [(40, 300, 20, 1, 0.5), (500, 150, 513, 30, 8.0), (3, 200, 8, 1, 50.0)])
def test_fusion_sums_its_components(n, b, feat, n_cls, spread):
    rng = np.random.default_rng(n + feat)
    ent, det = _world(rng, n, b, feat, n_cls, spread)
    ctx = F.farm_create(0)
    try:
        got = F.farm_associate(ctx, ent, det, 0.8, 0.9, 8)
    finally:
        F.farm_destroy(ctx)
    t = n + b
    # the components of the reported matches: smallest node of each
    label = np.arange(t)
    d, j = np.nonzero(got["match_idx"] >= 0)
    u, v = n + d, got["match_idx"][d, j]
    for _ in range(t):
        low = np.minimum(label[u], label[v])
        new = label.copy()
        np.minimum.at(new, u, low)
        np.minimum.at(new, v, low)
        if np.array_equal(new, label):
            break
        label = new
    w = np.concatenate([ent["w"], np.ones(b, np.float32)]).astype(np.float64)
    parent = np.arange(t)
    for c in np.unique(label):
        mem = np.flatnonzero(label == c)
        es = mem[mem < n]
        if es.size:
            parent[mem] = es[np.lexsort((es, -w[es]))[0]]
    np.testing.assert_array_equal(got["parent"], parent)
    mu = np.concatenate([ent["mu"], det["mu"]], axis=1).astype(np.float64)
    cv = np.concatenate([ent["cov"], det["cov"]], axis=1).astype(np.float64)
    ft = np.concatenate([ent["feat"], det["feat"]]).astype(np.float64)
    ia, ib = [0, 0, 0, 1, 1, 2], [0, 1, 2, 1, 2, 2]
    for g in range(t):
        mem = np.flatnonzero(parent == g)
        W = w[mem].sum() if mem.size else 0.0
        if W == 0.0:
            for k in ("mu", "cov"):
                assert not got[k][:, g].any()
            assert got["w"][g] == 0 and not got["feat"][g].any()
            continue
        m = (w[mem] * mu[:, mem]).sum(1) / W
        dm = mu[:, mem] - m[:, None]
        c = (w[mem] * (cv[:, mem] + dm[ia] * dm[ib])).sum(1) / W
        # FP32 sums of at most a few hundred members: relative errors of some 1e-5 of the summands
        assert got["w"][g] == W
        np.testing.assert_allclose(got["mu"][:, g], m, rtol=0, atol=2e-5)
        np.testing.assert_allclose(got["cov"][:, g], c, rtol=1e-4, atol=2e-6)
        np.testing.assert_allclose(got["feat"][g], (w[mem, None] * ft[mem]).sum(0) / W, rtol=0, atol=2e-6)
