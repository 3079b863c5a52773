"""What a training call leaves with its context: given back on release of a
scene and to an allocation that fails, and the next call trains as the first."""
import ctypes as C

import numpy as np
import pytest

F = pytest.importorskip("paper_2606_15476_gb300.farm")
pytestmark = pytest.mark.gpu


def _train(ctx, desc, rng):
    h, p, dim = 128, 64, desc.shape[1]
    g = np.random.default_rng(3)
    F.farm_mlp_set(ctx, *(g.standard_normal(s).astype(np.float32) / 8 for s in ((h, dim), (h,), (p, h), (p,))))
    b = 65536
    F.farm_mlp_train(ctx, 0, desc[:50], rng.integers(0, 50, b).astype(np.int32),
                     rng.integers(0, len(desc), b).astype(np.int32), rng.uniform(-1, 1, b).astype(np.float32),
                     epochs=1, batch=b)
    return F.farm_mlp_get(ctx, dim, h, p)          # (the loss is a sum in any order)


@pytest.mark.parametrize("how", ["release", "allocation"])
def test_training_memory_is_given_back(how):
    import torch
    rng = np.random.default_rng(5)
    desc = rng.standard_normal((300, 64)).astype(np.float32)
    ctx = F.farm_create(0)
    try:
        for sid in (0, 1):
            F.farm_memory_upload(ctx, sid, desc, np.zeros(300, np.int32), np.ones((6, 300), np.float32))
        first = _train(ctx, desc, np.random.default_rng(7))
        F.farm_sync(ctx)
        kept = torch.cuda.mem_get_info()[0]
        if how == "release":
            F.farm_memory_release(ctx, 1)
        else:
            some = torch.zeros(16, device="cuda")       # (2^40 rows: the call fails before it reads them)
            p = C.c_void_p(some.data_ptr())
            with pytest.raises(F.FarmError):
                F._ck(ctx, F._lib.farm_similarity(ctx, 0, 2 ** 40, p, F.PREC_FP32, p, F.PTR_DEVICE))
        # (the stacked activations alone: 131,072 rows x 128 hidden, two FP32 and two BF16 copies)
        assert torch.cuda.mem_get_info()[0] - kept > 131072 * 128 * 12
        again = _train(ctx, desc, np.random.default_rng(7))
        for a, b in zip(first, again):
            np.testing.assert_array_equal(a, b)
    finally:
        F.farm_destroy(ctx)
