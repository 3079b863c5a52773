"""Rank lists of scenes of more objects than the block-level select stages group
maxima for (8,192 groups of 32: 262,144 objects), whose best objects lie past
that prefix, above every staged maximum."""
import numpy as np
import pytest

F = pytest.importorskip("paper_2606_15476_gb300.farm")
pytestmark = pytest.mark.gpu

PREFIX = 8192 * 32
DIM = 64


def _unit(x):
    return x / np.linalg.norm(x, axis=1, keepdims=True)


def _world(n, queries, dim=DIM, seed=0):
    """Unit rows, queries, and per even query the objects planted for it past the
    prefix, best first: cosines 0.98, 0.96, ... (random ones stay below 0.75)."""
    rng = np.random.default_rng(n + queries + seed)
    desc = _unit(rng.standard_normal((n, dim)))
    q = _unit(rng.standard_normal((queries, dim)))
    per = min(8, (n - PREFIX) // max(1, (queries + 1) // 2)) if n - PREFIX > 1 else 1
    places = PREFIX + rng.permutation(n - PREFIX)
    plant, at = {}, 0
    for i in range(0, queries, 2):
        if at + per > len(places):
            break
        ids = places[at:at + per]
        at += per
        for j, o in enumerate(ids):
            c = 0.98 - 0.02 * j
            d = rng.standard_normal(dim)
            d -= (d @ q[i]) * q[i]
            desc[o] = c * q[i] + np.sqrt(1 - c * c) * d / np.linalg.norm(d)
        plant[i] = ids
    return desc.astype(np.float32), q.astype(np.float32), plant


def _ctx(k_max, k_anchor):
    p = F.farm_default_params()
    p.k_max, p.k_anchor = k_max, k_anchor
    return F.farm_create(0, None, p)


def _upload(ctx, desc):
    n = len(desc)
    rng = np.random.default_rng(1)
    F.farm_memory_upload(ctx, 0, desc, np.zeros(n, np.int32), rng.uniform(0.1, 5.0, (6, n)).astype(np.float32))


def _batch(ctx, q, precision, **kw):
    m = len(q)
    return F.farm_query_batch(ctx, np.zeros(m, np.int32), q, np.full(m, -1, np.int32), np.arange(m + 1, dtype=np.int32),
                              np.full(m, F.NEAR, np.int32), q, precision, **kw)


# (60 queries with as many landmark rows: the kernel for few rows; 700: the tiles)
@pytest.mark.parametrize("n", [PREFIX, PREFIX + 1, 270001, 300000])
@pytest.mark.parametrize("queries", [60, 700])
def test_fp32_lists_equal_a_stable_sort(n, queries):
    if n == PREFIX:      # (every maximum is staged)
        desc = _unit(np.random.default_rng(n).standard_normal((n, DIM))).astype(np.float32)
        q, plant = _unit(np.random.default_rng(n + 1).standard_normal((queries, DIM))).astype(np.float32), {}
    else:
        desc, q, plant = _world(n, queries)
        assert plant
    ctx = _ctx(60, 256)
    try:
        _upload(ctx, desc)
        h = _batch(ctx, q, F.PREC_FP32, fused=False)
        t, l = F.farm_candidates(ctx, h, queries, queries)
        assert t.shape[1] > 96 and l.shape[1] == 256
        for i in list(plant)[:8] + [1, 3, queries - 1]:
            cos = F.farm_similarity(ctx, 0, q[i:i + 1], n, F.PREC_FP32)[0]
            order = np.argsort(-cos, kind="stable")
            np.testing.assert_array_equal(t[i], order[:t.shape[1]])
            np.testing.assert_array_equal(l[i], order[:l.shape[1]])
            if i in plant:
                np.testing.assert_array_equal(t[i, :len(plant[i])], plant[i])
    finally:
        F.farm_destroy(ctx)


# (gaps of 0.02 between the planted cosines are far above BF16's and E4M3's errors
# over 64 random entries, about 2^-9 / 8 and 2^-4 / 8)
@pytest.mark.parametrize("precision", ["PREC_BF16", "PREC_FP8"])
@pytest.mark.parametrize("n", [PREFIX + 1, 300000])
def test_reduced_lists_begin_with_the_planted_objects(n, precision):
    desc, q, plant = _world(n, 60)
    ctx = _ctx(10, 16)
    try:
        _upload(ctx, desc)
        h = _batch(ctx, q, getattr(F, precision))
        t, l = F.farm_candidates(ctx, h, 60, 60)
        for i in range(60):
            for got in (t[i], l[i]):
                assert got.min() >= 0 and got.max() < n and len(set(got.tolist())) == len(got)
                cos = desc[got].astype(np.float64) @ q[i].astype(np.float64)
                # (FP32 dot products of rows normalised in FP32: within 4e-6 of these)
                assert (np.diff(cos) < 8e-6).all()
                if i in plant:
                    np.testing.assert_array_equal(got[:len(plant[i])], plant[i])
    finally:
        F.farm_destroy(ctx)


@pytest.mark.parametrize("n", [PREFIX + 1, 300000])
def test_two_channels_begin_with_the_planted_objects(n):
    """An object of rank j in both channels has the j-th largest fused score."""
    desc, q, plant = _world(n, 60)
    ctx = _ctx(8, 16)
    try:
        _upload(ctx, desc)
        F.farm_memory_add_space(ctx, 0, 1, desc)
        none = np.zeros((0, DIM), np.float32)
        h = F.farm_query_batch_rrf(ctx, 0, [(0, 1.0), (1, 1.0)], [q, q], np.full(60, -1, np.int32),
                                   np.zeros(61, np.int32), np.zeros(0, np.int32), [none, none])
        out = F.farm_topk(ctx, h, 8, 60)
        for i, ids in plant.items():
            np.testing.assert_array_equal(out["idx"][i, :len(ids)], ids)
    finally:
        F.farm_destroy(ctx)
