"""Batches of at most 128 rows over large scenes: stored rows up to 20 x 2^20 cosines
(short descriptors: 786,432 objects) and where a fused threshold would overflow,
fused beyond.  Both sides of each line give the forced routes' results."""
import numpy as np
import pytest

F = pytest.importorskip("paper_2606_15476_gb300.farm")
pytestmark = pytest.mark.gpu


# (104 x 201,000 and 786,432 / 786,433 objects: the lines; 128 rows of lists of 512
# over 300,001: beyond what the sample's keys refine, where the forced fused route
# leaves its rows to the exact fallback, whose FP32 sums are in another order)
@pytest.mark.parametrize("n,dim,queries,k_max", [(201000, 64, 52, 10), (202000, 64, 52, 10), (786432, 16, 3, 10),
                                                 (786433, 16, 3, 10), (300001, 32, 64, 60)])
def test_routes_agree(n, dim, queries, k_max):
    rng = np.random.default_rng(n)
    f = lambda *s: rng.standard_normal(s, dtype=np.float32)  # noqa: E731
    p = F.farm_default_params()
    p.k_max = k_max
    ctx = F.farm_create(0, None, p)
    try:
        F.farm_memory_upload(ctx, 0, f(n, dim), rng.integers(0, 50, n).astype(np.int32),
                             rng.uniform(0.1, 9.0, (6, n)).astype(np.float32))
        q, lm = f(queries, dim), f(queries, dim)
        got = []
        routes = [(None, False), (None, True), (False, False)] + ([(True, False)] if k_max == 10 else [])
        for fused, graph in routes:
            h = F.farm_query_batch(ctx, np.zeros(queries, np.int32), q, rng.integers(0, 1, queries).astype(np.int32),
                                   np.arange(queries + 1, dtype=np.int32), np.full(queries, F.NEAR, np.int32), lm,
                                   F.PREC_FP32, graph=graph, fused=fused)
            out = F.farm_topk(ctx, h, k_max, queries)
            got.append([out["idx"], out["score"], out["pred"], out["anchor"], *F.farm_candidates(ctx, h, queries, queries)])
    finally:
        F.farm_destroy(ctx)
    for g in got[1:]:
        for k, (a, b) in enumerate(zip(got[0], g)):
            np.testing.assert_array_equal(a, b)
