"""The single similarity problem on both sides of the few-row rule (97 to 128
rows: the few-row kernel from a third of the SMs in tiles of 128 objects on,
the CTA pairs below): the same products summed in the same order, so the
cosines and the rank lists agree bit for bit with the tile variants'."""
import numpy as np
import pytest

F = pytest.importorskip("paper_2606_15476_gb300.farm")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 300, 6400, 6401, 6529])
def test_cosines_agree(n):
    rng = np.random.default_rng(n)
    dim = 72
    d = rng.standard_normal((n, dim)).astype(np.float32)
    ctx = F.farm_create(0)
    try:
        F.farm_memory_upload(ctx, 0, d, np.zeros(n, np.int32), np.ones((6, n), np.float32))
        for rows in (96, 97, 128, 129):
            q = rng.standard_normal((rows, dim)).astype(np.float32)
            np.testing.assert_array_equal(F.farm_similarity(ctx, 0, q, n, F.PREC_FP32),
                                          F.farm_similarity_variant(ctx, 0, q, F.PREC_FP32, 1))
    finally:
        F.farm_destroy(ctx)
