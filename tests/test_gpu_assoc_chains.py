"""Components that grow through long chains of matches (each detection lies
between two entities of a row), whatever the order of the unions."""
import numpy as np
import pytest

F = pytest.importorskip("paper_2606_15476_gb300.farm")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,links,ordered", [(2, 1, True), (600, 599, True), (6000, 5999, False), (9000, 8200, False)])
def test_chains(n, links, ordered):
    rng = np.random.default_rng(n)
    place = np.arange(n) if ordered else rng.permutation(n)      # the chain's order against the numbers'
    mu = np.zeros((3, n), np.float32)
    mu[0, place] = np.arange(n)
    joined = np.sort(rng.permutation(n - 1)[:links])             # links i -- i + 1 of the chain
    dmu = np.zeros((3, links), np.float32)
    dmu[0] = joined + 0.5
    # deviation 0.2: H(0.5 apart) = sqrt(1 - exp(-0.25 / 0.32)) = 0.74, H(1.5 apart) > 0.999
    cov = lambda k: np.repeat(np.float32([[0.04], [0], [0], [0.04], [0], [0.04]]), k, 1)  # noqa: E731
    one = lambda k: np.ones((k, 1), np.float32)  # noqa: E731
    w = rng.permutation(n).astype(np.float32)
    ent = dict(mu=mu, cov=cov(n), feat=one(n), w=w, active=np.ones(n, np.int32))
    det = dict(mu=dmu, cov=cov(links), feat=one(links))
    ctx = F.farm_create(0)
    try:
        runs = [F.farm_associate(ctx, ent, det, 0.5, 0.9, 4) for _ in range(3)]
    finally:
        F.farm_destroy(ctx)
    cut = np.ones(n, bool)                                       # the chain's places that start a component
    cut[joined + 1] = False
    comp = np.cumsum(cut) - 1
    best = np.full(comp[-1] + 1, -1)
    for i in np.argsort(w[place]):                               # the heaviest entity of each comes last
        best[comp[i]] = place[i]
    want = np.empty(n + links, np.int64)
    want[place] = best[comp]
    want[n:] = best[comp[joined]]
    for got in runs:
        assert (got["match_cnt"] == 2).all()
        np.testing.assert_array_equal(got["parent"], want)
