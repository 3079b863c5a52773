"""The sixteen-warp epilogue of the BF16 similarity over short rows (tile
variants 0 and 2) against the four-warp one (variant 1, and rows past the
rule's bound): every variant computes each cosine with the same products in
the same order, so cosines and rank lists agree bit for bit."""
import numpy as np
import pytest

import synth

F = pytest.importorskip("paper_2606_15476_gb300.farm")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim", [64, 448, 512, 520])
@pytest.mark.parametrize("rows,n", [(1, 255), (129, 257), (300, 8193)])
def test_cosines_agree(dim, rows, n):
    rng = np.random.default_rng(dim + n)
    d = rng.standard_normal((n, dim)).astype(np.float32)
    q = rng.standard_normal((rows, dim)).astype(np.float32)
    ctx = F.farm_create(0)
    try:
        F.farm_memory_upload(ctx, 0, d, np.zeros(n, np.int32), np.ones((6, n), np.float32))
        ref = F.farm_similarity_variant(ctx, 0, q, F.PREC_BF16, 1)
        for v in (0, 2):
            np.testing.assert_array_equal(F.farm_similarity_variant(ctx, 0, q, F.PREC_BF16, v), ref)
    finally:
        F.farm_destroy(ctx)


@pytest.mark.parametrize("n", [700, 2500, 8300, 65537])     # groups of 8 and of 32; the last takes the two-pass form
def test_learned_lists_agree(n):
    dim = 64
    sc = synth.make_scene(9, n, dim, extent=(60.0, 60.0, 5.0), n_classes=max(16, n // 50), n_views=1)
    qb = synth.make_queries(10, sc, 70, m_choices=(1, 2))
    rng = np.random.default_rng(5)
    ctx = F.farm_create(0)
    try:
        F.farm_memory_upload(ctx, 0, sc.desc, sc.cls, sc.box, sc.views)
        F.farm_mlp_set(ctx, *[(rng.standard_normal(s) / np.sqrt(s[-1])).astype(np.float32)
                              for s in ((64, dim), (64,), (128, 64), (128,))])
        got = []
        for v in (1, 0, 2):
            F.farm_sim_variant_pin(ctx, v)
            h = F.farm_query_batch(ctx, qb.scene_of_q, qb.tgt_emb, qb.tgt_cls, qb.c_off, qb.c_pred, qb.c_emb,
                                   F.PREC_LEARNED)
            got.append(F.farm_candidates(ctx, h, qb.n_q, qb.n_c))
        for t, lm in got[1:]:
            np.testing.assert_array_equal(t, got[0][0])
            np.testing.assert_array_equal(lm, got[0][1])
        assert F.farm_select_fallbacks(ctx) == 0
    finally:
        F.farm_destroy(ctx)
