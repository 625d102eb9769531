"""The sorted read-out: a rank count for small pools, a radix sort for larger ones.
Both give the cells of the unsorted read-out in lexicographic order of the indices."""
import ctypes

import numpy as np
import pytest

from paper_2508_13986_gb300 import gbees
from paper_2508_13986_gb300 import workloads as W

pytestmark = pytest.mark.gpu


# pools (active cells and halo) below, around and above the 2^14 entries of the rank
# count; widths of the index ranges from one value (no pass at all in that field) up
@pytest.mark.parametrize("n,count,radius", [(1, 1, 5), (1, 16000, 40000), (2, 3000, 2000), (2, 60000, 30000),
                                            (3, 2300, 400), (3, 2400, 1), (3, 30000, 500), (4, 9000, 60),
                                            (5, 20000, 12), (6, 1200, 200), (6, 40000, 5)])
@pytest.mark.parametrize("prec", [gbees.GBEES_FP64, gbees.GBEES_FP32])
def test_sorted_read_out_is_the_lexicographic_order(n, count, radius, prec):
    idx, p = W.random_cells(n, count, min(radius, 500 if n > 3 else radius), seed=n + count)
    idx[:, 0] += 3 - radius // 2
    cfg = gbees.make_config(n, gbees.GBEES_DYN_CONSTANT, [0.5] * n, [0.25] * n, [0.0] * n, 1e-3, precision=prec,
                            max_cells=1 << (24 if n > 4 else 22))
    g = gbees.Grid(cfg)
    g.init_cells(idx, p)
    ui, up = g.read_cells(sorted_=False)
    si, sp = g.read_cells(sorted_=True)
    order = np.lexsort(ui.T[::-1])
    assert np.array_equal(si, ui[order]) and np.array_equal(sp, up[order])
    # a buffer that is too small gets the first cells and EINVAL
    cap = max(1, idx.shape[0] // 3)
    ci, cp, cnt = np.full((cap, n), -9, dtype=np.int32), np.zeros(cap), ctypes.c_int64()
    rc, cnt = gbees.gbees_read_cells(g.ctx, ci, cp, True)
    assert cnt == idx.shape[0]
    assert rc == (gbees.GBEES_EINVAL if cap < cnt else gbees.GBEES_OK)
    assert np.array_equal(ci, si[:cap]) and np.array_equal(cp, sp[:cap])
    # the read-out leaves the grid as it was
    st = g.propagate(0.1)
    h = gbees.Grid(cfg)
    h.init_cells(idx, p)
    assert h.propagate(0.1) == st
    for a, b in zip(g.read_cells(), h.read_cells()):
        assert np.array_equal(a, b)
