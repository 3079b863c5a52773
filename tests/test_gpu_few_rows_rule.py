"""The FP32-accurate tile configurations on both sides of the rules that choose
them (65 to 128 rows: 128 x 128 tiles on at most half of the SMs, else the
few-row kernel; more rows: those on at most a quarter, 128 x 256 tiles where
they save enough waves, else the CTA pairs): the same products summed in the
same order, so the cosines of whichever is taken, odd leading dimensions
included, and the rank lists of batches agree bit for bit with a pinned
variant's."""
import numpy as np
import pytest

import synth

F = pytest.importorskip("paper_2606_15476_gb300.farm")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 127, 300, 2001, 4864, 9728, 9729, 19601])
@pytest.mark.parametrize("dim", [72, 1000])
def test_cosines_agree(n, dim):
    rng = np.random.default_rng(n)
    d = rng.standard_normal((n, dim)).astype(np.float32)
    ctx = F.farm_create(0)
    try:
        F.farm_memory_upload(ctx, 0, d, np.zeros(n, np.int32), np.ones((6, n), np.float32))
        for rows in (64, 65, 128, 129, 257, 300, 701):
            q = rng.standard_normal((rows, dim)).astype(np.float32)
            np.testing.assert_array_equal(F.farm_similarity(ctx, 0, q, n, F.PREC_FP32),
                                          F.farm_similarity_variant(ctx, 0, q, F.PREC_FP32, 2))
    finally:
        F.farm_destroy(ctx)


@pytest.mark.parametrize("n,n_q", [(700, 30), (9728, 30), (9729, 30)])
def test_batches_agree(n, n_q):
    sc = synth.make_scene(90, n, 64, extent=(30.0, 30.0, 4.0), n_classes=20, n_views=2)
    qb = synth.make_queries(91, sc, n_q, m_choices=(2,))        # 90 rows
    ctx = F.farm_create(0)
    try:
        F.farm_memory_upload(ctx, 0, sc.desc, sc.cls, sc.box, sc.views)
        got = []
        for pin, graph in ((-1, False), (-1, True), (2, False)):
            F.farm_sim_variant_pin(ctx, pin)
            h = F.farm_query_batch(ctx, np.zeros(n_q, np.int32), qb.tgt_emb, qb.tgt_cls, qb.c_off, qb.c_pred, qb.c_emb,
                                   F.PREC_FP32, graph=graph, fused=False)
            out = F.farm_topk(ctx, h, 10, n_q)
            got.append([out["idx"], out["score"], out["pred"], out["anchor"], *F.farm_candidates(ctx, h, qb.n_q, qb.n_c)])
        for g in got[1:]:
            for a, b in zip(got[0], g):
                np.testing.assert_array_equal(a, b)
    finally:
        F.farm_destroy(ctx)
