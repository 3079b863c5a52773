"""E4M3 copies made by the normalising pass, for the scene's rows and the
queries': FP8 cosines against the same quantisation done with PyTorch, at widths
that take four entries at a time and widths that do not, with a zero tail up to
the padded width.  Bound: 16 FP32 roundings of sums below 1, and one entry per
pair whose quotient rounds the other way (a step of 2^-4 of at most
max|x| max|y|); a wrong scale or byte is off by far more."""
import numpy as np
import pytest
import torch

F = pytest.importorskip("paper_2606_15476_gb300.farm")
pytestmark = pytest.mark.gpu


def _quantised(x):
    x = torch.from_numpy(x)
    u = x / torch.linalg.vector_norm(x.double(), dim=1, keepdim=True).float()
    sc = u.abs().amax(1, keepdim=True) / 448.0
    return (u / sc).to(torch.float8_e4m3fn).double() * sc.double(), u.abs().amax(1).double()


@pytest.mark.parametrize("dim", [1, 3, 66, 127, 128, 130, 1000, 1152])
def test_cosines_of_quantised_rows(dim):
    rng = np.random.default_rng(dim)
    d = rng.standard_normal((300, dim)).astype(np.float32)
    q = (rng.standard_normal((37, dim)) * 10.0 ** rng.integers(-6, 6, (37, 1))).astype(np.float32)
    ctx = F.farm_create(0)
    try:
        F.farm_memory_upload(ctx, 0, d, np.zeros(300, np.int32), np.ones((6, 300), np.float32))
        got = F.farm_similarity(ctx, 0, q, 300, F.PREC_FP8)
    finally:
        F.farm_destroy(ctx)
    (qq, qm), (dd, dm) = _quantised(q), _quantised(d)
    bound = 16 * 2.0 ** -24 + 2.0 ** -4 * qm[:, None] * dm[None, :]
    assert ((torch.from_numpy(got).double() - qq @ dd.T).abs() <= bound).all()
