"""The grouped FP32 rescore (four rows per block, candidates of their union
loaded once) against the row-per-block one: a large batch takes the first, the
same queries in small batches the second, and every list must agree entry for
entry.  Two scenes in one batch, so that some blocks hold rows of both."""
import numpy as np
import pytest

import synth

F = pytest.importorskip("paper_2606_15476_gb300.farm")
pytestmark = pytest.mark.gpu

GROUP_FROM = 2048       # rows of a launch from which blocks take four


def _batch(F, ctx, qb, prec):
    h = F.farm_query_batch(ctx, qb.scene_of_q, qb.tgt_emb, qb.tgt_cls, qb.c_off, qb.c_pred, qb.c_emb, prec)
    out = F.farm_topk(ctx, h, 10, qb.n_q)
    t, lm = F.farm_candidates(ctx, h, qb.n_q, qb.n_c)
    return [out["idx"], out["score"], out["pred"], out["anchor"], t], lm


@pytest.mark.parametrize("dim,prec,ns", [(72, "bf16", (16400, 17000)), (72, "fp8", (16400, 17000)),
                                         (1152, "bf16", (16400, 16500)), (100, "learned", (700, 1500)),
                                         (2048, "learned", (900, 600)), (2100, "learned", (900, 600))])
def test_groups_equal_single_rows(dim, prec, ns):
    code = {"bf16": F.PREC_BF16, "fp8": F.PREC_FP8, "learned": F.PREC_LEARNED}[prec]
    scenes = [synth.make_scene(50 + i, n, dim, extent=(40.0, 40.0, 4.0), n_classes=60, n_views=2, distractor_classes=4,
                               distractor_frac=0.3) for i, n in enumerate(ns)]
    parts = [synth.make_queries(60 + i, s, 551 + 2 * i, m_choices=(0, 1, 2, 3), distractor_classes=4,
                                distractor_target_frac=0.5, scene_id=i) for i, s in enumerate(scenes)]
    from synth.scenes import concat_batches
    qb = concat_batches(parts).subset(np.random.default_rng(3).permutation(sum(p.n_q for p in parts)))
    assert qb.n_q + qb.n_c >= GROUP_FROM
    ctx = F.farm_create(0)
    try:
        for i, s in enumerate(scenes):
            F.farm_memory_upload(ctx, i, s.desc, s.cls, s.box, s.views)
        if prec == "learned":
            rng = np.random.default_rng(5)
            F.farm_mlp_set(ctx, *[(rng.standard_normal(sh) / np.sqrt(sh[-1])).astype(np.float32)
                                  for sh in ((64, dim), (64,), (64, 64), (64,))])
        whole, lm = _batch(F, ctx, qb, code)
        step = 300                       # at most 300 + 900 rows
        for q0 in range(0, qb.n_q, step):
            qs = np.arange(q0, min(qb.n_q, q0 + step))
            sub = qb.subset(qs)
            assert sub.n_q + sub.n_c < GROUP_FROM
            got, l2 = _batch(F, ctx, sub, code)
            for a, b in zip(whole, got):
                np.testing.assert_array_equal(a[qs], b)
            np.testing.assert_array_equal(lm[qb.c_off[q0]:qb.c_off[qs[-1] + 1]], l2)
    finally:
        F.farm_destroy(ctx)
