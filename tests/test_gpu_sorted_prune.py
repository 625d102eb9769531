"""The sorted prune of a large grid against the plain one of a small grid.

The graph and direct paths sort the survivors, move them in that order with their links
and rehash them in one pass; the persistent kernel compacts them in place. The order
decides no result, so both end bit for bit alike. Sizes: pools at the edges of a warp, of
a block and of the sort's tiles, and one whose sort takes several tiles per block."""
import numpy as np
import pytest

from paper_2508_13986_gb300 import gbees
from paper_2508_13986_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _run(n, prec, mode, idx, p):
    rng = np.random.Generator(np.random.PCG64(90 + n))
    a = rng.uniform(-1.0, 1.0, n * n + n)
    cfg = gbees.make_config(n, gbees.GBEES_DYN_LINEAR, a, [0.5] * n, [0.1] * n, 1e-3, 0.9, 1, prec,
                            max_cells=1 << 21, launch_mode=mode)
    g = gbees.Grid(cfg)
    g.init_cells(idx, p)
    s = g.propagate(0.02)
    out = (*g.read_cells(), *g.moments(), (s.steps, s.cell_updates, s.n_cells, s.n_pool, s.t, s.norm))
    g.close()
    return out


@pytest.mark.parametrize("prec", [gbees.GBEES_FP64, gbees.GBEES_FP32])
@pytest.mark.parametrize("n,count,radius,mode", [
    (1, 1, 1, gbees.GBEES_LAUNCH_GRAPH), (1, 31, 15, gbees.GBEES_LAUNCH_GRAPH), (1, 255, 127, gbees.GBEES_LAUNCH_GRAPH),
    (1, 1023, 511, gbees.GBEES_LAUNCH_GRAPH), (2, 1025, 16, gbees.GBEES_LAUNCH_GRAPH),
    (3, 60000, 40, gbees.GBEES_LAUNCH_DIRECT)])
def test_sorted_prune_equals_the_plain_one(n, count, radius, mode, prec):
    idx, p = W.random_cells(n, count, radius, seed=3 + n)
    got = _run(n, prec, mode, idx, p)
    ref = _run(n, prec, gbees.GBEES_LAUNCH_PERSISTENT, idx, p)
    assert got[4] == ref[4]
    for x, y in zip(got[:4], ref[:4]):
        assert np.array_equal(x, y)
