"""Calls that fail for want of device memory (sizes far beyond the card's) after
they have given up arrays that a recorded graph batch reads: the next call of
that batch must not be replayed over them."""
import ctypes as C

import numpy as np
import pytest

import synth

F = pytest.importorskip("paper_2606_15476_gb300.farm")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def world():
    return synth.make_scene(5, 700, 64, extent=(12.0, 12.0, 3.0), n_classes=9, n_views=2)


def _ask(ctx, qb):
    h = F.farm_query_batch(ctx, qb.scene_of_q, qb.tgt_emb, qb.tgt_cls, qb.c_off, qb.c_pred, qb.c_emb, F.PREC_FP32, graph=True)
    out = F.farm_topk(ctx, h, 10, qb.n_q)
    return [out[k] for k in ("idx", "score", "pred", "anchor")]


def _recorded(ctx, s):
    F.farm_memory_upload(ctx, 0, s.desc, s.cls, s.box, s.views)
    qb = synth.make_queries(6, s, 150, m_choices=(1, 2))
    for _ in range(4):            # tuned, captured for both slots of the host rows, replayed
        first = _ask(ctx, qb)
    return qb, first


def test_failed_upload_over_a_recorded_scene(world):
    import torch
    ctx = F.farm_create(0)
    try:
        qb, first = _recorded(ctx, world)
        some = torch.zeros(16, device="cuda")           # (the call fails before it reads them)
        p = C.c_void_p(some.data_ptr())
        with pytest.raises(F.FarmError):
            F._ck(ctx, F._lib.farm_memory_upload(ctx, 0, 2 ** 31 - 1, 8192, p, p, p, 0, None, F.PTR_DEVICE))
        with pytest.raises(F.FarmError, match="unknown scene"):
            _ask(ctx, qb)
        F.farm_memory_upload(ctx, 0, world.desc, world.cls, world.box, world.views)
        for _ in range(3):
            for a, b in zip(first, _ask(ctx, qb)):
                np.testing.assert_array_equal(a, b)
    finally:
        F.farm_destroy(ctx)


def test_failed_growth_of_a_recorded_buffer(world):
    import torch
    ctx = F.farm_create(0)
    try:
        qb, first = _recorded(ctx, world)
        some = torch.zeros(16, device="cuda")
        p = C.c_void_p(some.data_ptr())
        with pytest.raises(F.FarmError):                # (2^40 rows: the operand rows' buffer is given up, not had)
            F._ck(ctx, F._lib.farm_similarity(ctx, 0, 2 ** 40, p, F.PREC_FP32, p, F.PTR_DEVICE))
        for _ in range(3):
            for a, b in zip(first, _ask(ctx, qb)):
                np.testing.assert_array_equal(a, b)
    finally:
        F.farm_destroy(ctx)
