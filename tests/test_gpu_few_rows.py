"""The few-row similarity (batches of at most 128 query rows, the operands'
roles exchanged) against the tile variants: the same products summed in the
same order, so cosines, group maxima and rank lists agree bit for bit."""
import numpy as np
import pytest

import synth
from synth.scenes import concat_batches

F = pytest.importorskip("paper_2606_15476_gb300.farm")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim", [40, 1152])
@pytest.mark.parametrize("n", [1, 127, 129, 8192])
def test_cosines_agree(dim, n):
    rng = np.random.default_rng(dim + n)
    d = rng.standard_normal((n, dim)).astype(np.float32)
    ctx = F.farm_create(0)
    try:
        F.farm_memory_upload(ctx, 0, d, np.zeros(n, np.int32), np.ones((6, n), np.float32))
        for rows in (1, 16, 17, 33, 64, 65, 128, 129):       # the last takes the CTA pairs
            q = rng.standard_normal((rows, dim)).astype(np.float32)
            np.testing.assert_array_equal(F.farm_similarity(ctx, 0, q, n, F.PREC_FP32),
                                          F.farm_similarity_variant(ctx, 0, q, F.PREC_FP32, 1))
    finally:
        F.farm_destroy(ctx)


@pytest.mark.parametrize("ns,per", [((1,), 1), ((57, 2049, 8191), 9), ((8193, 40, 33000), 14), ((12288,), 25)])
def test_batches_agree(ns, per):
    scenes = [synth.make_scene(70 + i, n, 64, extent=(30.0, 30.0, 4.0), n_classes=20, n_views=2)
              for i, n in enumerate(ns)]
    qb = concat_batches([synth.make_queries(80 + i, s, per, m_choices=(0, 1, 2), scene_id=i)
                         for i, s in enumerate(scenes)])
    ctx = F.farm_create(0)
    try:
        for i, s in enumerate(scenes):
            F.farm_memory_upload(ctx, i, s.desc, s.cls, s.box, s.views)
        got = []
        for pin, fused, graph in ((-1, None, False), (-1, None, True), (-1, False, False), (1, False, False),
                                  (0, True, False)):
            F.farm_sim_variant_pin(ctx, pin)
            h = F.farm_query_batch(ctx, qb.scene_of_q, qb.tgt_emb, qb.tgt_cls, qb.c_off, qb.c_pred, qb.c_emb,
                                   F.PREC_FP32, graph=graph, fused=fused)
            k = min(10, min(ns))
            out = F.farm_topk(ctx, h, k, qb.n_q)
            got.append([out["idx"], out["score"], out["pred"], out["anchor"], *F.farm_candidates(ctx, h, qb.n_q, qb.n_c)])
        for g in got[1:]:
            for a, b in zip(got[0], g):
                np.testing.assert_array_equal(a, b)
    finally:
        F.farm_destroy(ctx)
