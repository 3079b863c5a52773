"""The block-level rank select (value bins for the bound and for the ranks) and
the warp-level one of small scenes' rows, against a stable sort of the same
cosines: list lengths on both sides of its routes, rows with every value
shared by several objects, short and long rows, launches on both sides of the
bound from which small rows take a warp each."""
import numpy as np
import pytest

F = pytest.importorskip("paper_2606_15476_gb300.farm")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [300, 2048, 2049, 8192, 40000])
@pytest.mark.parametrize("k_max,k_anchor,queries", [(1, 1, 20), (10, 16, 20), (60, 256, 20), (10, 16, 700), (60, 129, 650)])
@pytest.mark.parametrize("copies", [1, 3])
def test_lists_equal_a_stable_sort(n, k_max, k_anchor, queries, copies):
    rng = np.random.default_rng(n + k_max + queries)
    dim = 16
    desc = rng.standard_normal((n, dim)).astype(np.float32)
    if copies > 1:
        desc = desc[rng.integers(0, max(1, n // copies), n)]
    p = F.farm_default_params()
    p.k_max, p.k_anchor = k_max, k_anchor
    q = rng.standard_normal((queries, dim)).astype(np.float32)
    lm = rng.standard_normal((queries, dim)).astype(np.float32)
    ctx = F.farm_create(0, None, p)
    try:
        F.farm_memory_upload(ctx, 0, desc, rng.integers(0, 5, n).astype(np.int32),
                             rng.uniform(0.1, 5.0, (6, n)).astype(np.float32))
        h = F.farm_query_batch(ctx, np.zeros(queries, np.int32), q, np.full(queries, -1, np.int32),
                               np.arange(queries + 1, dtype=np.int32), np.full(queries, F.NEAR, np.int32), lm,
                               F.PREC_FP32, fused=False)
        t, l = F.farm_candidates(ctx, h, queries, queries)
        for rows, got in ((q, t), (lm, l)):
            for i in rng.choice(queries, 20, replace=False):
                cos = F.farm_similarity(ctx, 0, rows[i:i + 1], n, F.PREC_FP32)[0]
                np.testing.assert_array_equal(got[i], np.argsort(-cos, kind="stable")[:got.shape[1]])
    finally:
        F.farm_destroy(ctx)
