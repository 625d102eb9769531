"""The storage order of the pool decides no result: sorted in any of the orders, or sorted
between prunes as a large pool that has grown is, every run ends bit for bit as one that
never sorts."""
import numpy as np
import pytest

from paper_2508_13986_gb300 import gbees
from paper_2508_13986_gb300 import workloads as W

pytestmark = pytest.mark.gpu

PREC = pytest.mark.parametrize("prec", [gbees.GBEES_FP64, gbees.GBEES_FP32])


def _results(g, stats):
    out = (*g.read_cells(), *g.moments(), (stats.steps, stats.cell_updates, stats.n_cells, stats.n_pool, stats.t,
                                           stats.norm))
    launches = g.profile()["total_launches"]
    g.close()
    return out, launches


def _same(got, ref):
    assert got[4] == ref[4]
    for x, y in zip(got[:4], ref[:4]):
        assert np.array_equal(x, y)


@PREC
@pytest.mark.parametrize("n,h,mode", [(6, 0.33, gbees.GBEES_LAUNCH_GRAPH), (5, 0.2, gbees.GBEES_LAUNCH_GRAPH),
                                      (6, 0.33, gbees.GBEES_LAUNCH_DIRECT)])
def test_a_pool_sorted_between_prunes_gives_the_same(n, h, mode, prec):
    """2.7 to 3.5e6 entries, a third to two thirds of them out of order after the first
    step, no prune, 60 steps to go: sorted at once (seen from the launches), with the
    marks of what is complete and the values kept."""
    mean = np.full(n, 4.0)
    mean[0] += 0.5
    runs = {}
    for order in (gbees.GBEES_ORDER_KEY, gbees.GBEES_ORDER_NONE):
        cfg = gbees.make_config(n, gbees.GBEES_DYN_LORENZ96, [4.0], [h] * n, mean, 1e-6, 0.9, 0, prec,
                                max_cells=1 << 24, launch_mode=mode, storage_order=order)
        g = gbees.Grid(cfg)
        g.init_gaussian(mean, 0.25 * np.eye(n))
        g.propagate(0.002)
        st = g.propagate(0.24)
        runs[order] = _results(g, st)
    (got, sorted_launches), (ref, launches) = runs[gbees.GBEES_ORDER_KEY], runs[gbees.GBEES_ORDER_NONE]
    _same(got, ref)
    assert got[4][3] > 1 << 21
    if mode == gbees.GBEES_LAUNCH_GRAPH:  # (direct launches do nothing when nothing is due)
        assert sorted_launches > launches


@PREC
@pytest.mark.parametrize("order", [gbees.GBEES_ORDER_MORTON, gbees.GBEES_ORDER_KEY_MIXED, gbees.GBEES_ORDER_ROW_MORTON])
@pytest.mark.parametrize("n,count,radius", [(1, 300, 200), (2, 1025, 16), (3, 4000, 14), (6, 1500, 3)])
def test_prunes_in_every_order_give_the_same(n, count, radius, order, prec):
    idx, p = W.random_cells(n, count, radius, seed=5 + n)
    a = np.random.Generator(np.random.PCG64(60 + n)).uniform(-1.0, 1.0, n * n + n)
    runs = []
    for o in (order, gbees.GBEES_ORDER_NONE):
        cfg = gbees.make_config(n, gbees.GBEES_DYN_LINEAR, a, [0.5] * n, [0.1] * n, 1e-3, 0.9, 2, prec,
                                max_cells=1 << 21, launch_mode=gbees.GBEES_LAUNCH_GRAPH, storage_order=o)
        g = gbees.Grid(cfg)
        g.init_cells(idx, p)
        runs.append(_results(g, g.propagate(0.05))[0])
    _same(*runs)
