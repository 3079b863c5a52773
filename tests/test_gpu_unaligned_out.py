"""Cosines into device memory that starts on no 16-byte boundary (part of a larger
array), rows of a multiple of four and of other lengths."""
import numpy as np
import pytest

F = pytest.importorskip("paper_2606_15476_gb300.farm")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["PREC_FP32", "PREC_BF16", "PREC_FP8", "PREC_FP32_SIMT"])
@pytest.mark.parametrize("n", [512, 1301])
def test_cosines_anywhere(n, precision):
    import torch
    prec, rng = getattr(F, precision), np.random.default_rng(n)
    desc = rng.standard_normal((n, 64)).astype(np.float32)
    ctx = F.farm_create(0)
    try:
        F.farm_memory_upload(ctx, 0, desc, np.zeros(n, np.int32), np.ones((6, n), np.float32))
        for rows in (20, 100, 300, 1100):
            q = torch.from_numpy(rng.standard_normal((rows, 64)).astype(np.float32)).cuda()
            want = torch.zeros(rows, n, device="cuda")
            torch.cuda.synchronize()                  # (the context has a stream of its own)
            F.farm_similarity(ctx, 0, q, n, prec, out=want)
            F.farm_sync(ctx)
            for off in (1, 2, 3):
                buf = torch.full((rows * n + 8,), -9.0, device="cuda")
                torch.cuda.synchronize()
                F.farm_similarity(ctx, 0, q, n, prec, out=buf[off:off + rows * n].view(rows, n))
                F.farm_sync(ctx)
                assert torch.equal(buf[off:off + rows * n].view(rows, n), want)
                assert (buf[:off] == -9).all() and (buf[off + rows * n:] == -9).all()
    finally:
        F.farm_destroy(ctx)
