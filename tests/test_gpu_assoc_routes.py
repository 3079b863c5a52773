"""The association's routes above the size from which it emits (6 M cosines):
lists only, lists of which some overflow their buffer (their rows are then
computed and stored), and every row stored because a sample says that most
lists would overflow; padded and long feature lengths.  Against calls of 100
detections, which store their rows (a detection's matches depend on it and the
entities alone)."""
import numpy as np
import pytest

F = pytest.importorskip("paper_2606_15476_gb300.farm")
pytestmark = pytest.mark.gpu


def _world(rng, n, b, feat, alike, n_cls):
    """Entities 0 .. alike - 1 of one class, the others of n_cls - 1; detections
    re-observe entities drawn from all of them."""
    unit = lambda x: x / np.linalg.norm(x, axis=1, keepdims=True)  # noqa: E731
    cen = unit(rng.standard_normal((n_cls, feat)))
    cls = np.where(np.arange(n) < alike, 0, rng.integers(1, n_cls, n))
    src = rng.integers(0, n, b)
    mu, var = rng.uniform(0, 30, (3, n)), rng.uniform(0.01, 0.1, (3, n))

    def cov(v):
        z = np.zeros(v.shape[1])
        return np.stack([v[0], z, z, v[1], z, v[2]]).astype(np.float32)
    f32 = lambda x: np.ascontiguousarray(x, dtype=np.float32)  # noqa: E731
    ent = dict(mu=f32(mu), cov=cov(var), feat=f32(unit(cen[cls] + 0.01 * rng.standard_normal((n, feat)))),
               w=rng.integers(0, 9, n).astype(np.float32), active=(rng.uniform(size=n) > 0.1).astype(np.int32))
    det = dict(mu=f32(mu[:, src] + 0.05 * rng.standard_normal((3, b))), cov=cov(var[:, src]),
               feat=f32(unit(cen[cls[src]] + 0.01 * rng.standard_normal((b, feat)))))
    return ent, det


# mean list against 7/8 of the buffer's 2,048 (1,500 for 3,000 entities): far
# below; a fifth of the lists over 2,048, mean 540; mean 2,250 and all entities
@pytest.mark.parametrize("n,b,feat,alike,n_cls,tau", [
    (9000, 700, 7, 40, 200, 0.99), (9000, 705, 20, 30, 300, 0.8), (3001, 2100, 256, 30, 100, 0.8),
    (12000, 530, 500, 2500, 400, 0.8), (12001, 530, 256, 2500, 400, 0.8), (70000, 129, 64, 2049, 400, 0.8),
    (9000, 720, 64, 10, 5, 0.8), (8000, 800, 20, 100, 50, -1.0)])
def test_matches_equal_those_of_small_calls(n, b, feat, alike, n_cls, tau):
    assert n * b >= 6 << 20
    ent, det = _world(np.random.default_rng(n + feat), n, b, feat, alike, n_cls)
    ctx = F.farm_create(0)
    try:
        runs = [F.farm_associate(ctx, ent, det, tau, 0.9, 8) for _ in range(2)]
        for d0 in range(0, b, 100):
            part = {k: np.ascontiguousarray(v[d0:d0 + 100] if k == "feat" else v[:, d0:d0 + 100]) for k, v in det.items()}
            got = F.farm_associate(ctx, ent, part, tau, 0.9, 8)
            for whole in runs:
                for k in ("match_cnt", "match_idx", "match_h"):
                    np.testing.assert_array_equal(whole[k][d0:d0 + 100], got[k])
    finally:
        F.farm_destroy(ctx)
