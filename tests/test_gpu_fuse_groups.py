"""Exact ranks of the channel fusion at the edges of its group lists: the
groups of a similarity row that can hold entries above a probe are listed
2,048 at a time and read four entries at a time, so the sizes here leave every
remainder of four in the last group, of both group widths, and
end just at, below and past one stretch of the list (2,048 groups of 32).
"""
import numpy as np
import pytest

from oracle import parity
from test_gpu_rrf import F, ctx, _case, _run, _upload  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [257, 1022, 1023, 2047, 2048, 2049, 65535, 65536, 65537, 65570])
def test_group_list_edges(F, ctx, n):  # noqa: F811
    sc, sp, qb, cq = _case(1700 + n % 97, n, 64, (32, 96), 12, (60.0, 60.0, 6.0), n_classes=max(16, n // 50))
    _upload(F, ctx, 74, sc, sp)
    _, out = _run(F, ctx, 74, qb, cq)
    rep = parity.check_topk_mc(sc, sp.desc, qb, cq, 10, out["idx"], out["score"], out["pred"], out["anchor"])
    assert rep.ok(), rep.summary()
    _, again = _run(F, ctx, 74, qb, cq)     # (the lists' order is not fixed; the counts are)
    assert np.array_equal(out["idx"], again["idx"]) and np.array_equal(out["score"], again["score"])
