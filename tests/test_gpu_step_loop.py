"""The step loop of a small grid against the kernels of a large one.

The persistent kernel's phases are forms of their own (requests of the growing
cells in a list of fixed size per block, halo cells claimed in one phase and
completed in the next, fluxes at new entries in closed form). Both launch modes
perform the same IEEE operations on every density and sum exactly, so they end
bit for bit alike, on any number of blocks."""
import numpy as np
import pytest

from paper_2508_13986_gb300 import gbees
from paper_2508_13986_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _run(n, prec, mode, blocks, idx, p, prune_interval):
    rng = np.random.Generator(np.random.PCG64(40 + n))
    a = rng.uniform(-1.0, 1.0, n * n + n)
    cfg = gbees.make_config(n, gbees.GBEES_DYN_LINEAR, a, [0.5] * n, [0.1] * n, 1e-3, 0.9, prune_interval, prec,
                            max_cells=1 << 22, launch_mode=mode)
    g = gbees.Grid(cfg)
    assert gbees.gbees_set_persist_blocks(g.ctx, blocks) == gbees.GBEES_OK
    g.init_cells(idx, p)
    st = []
    for t in (0.02, 0.05):  # two launches: nothing of the first may leak into the second
        s = g.propagate(t)
        st.append((s.steps, s.cell_updates, s.n_cells, s.t, s.norm))
    out = (*g.read_cells(), *g.moments(), st)
    g.close()
    return out


@pytest.mark.parametrize("prec", [gbees.GBEES_FP64, gbees.GBEES_FP32])
@pytest.mark.parametrize("n,count,radius", [(1, 300, 400), (2, 5000, 60), (3, 6000, 16), (4, 4000, 6), (5, 2000, 4),
                                            (6, 1500, 3)])
def test_step_loop_equals_graph(n, count, radius, prec):
    """Random ragged sets (every cell grows, most of its neighbours missing): on one
    block the grow asks for more than its list of 1024 holds; 3 and 152 blocks
    leave it short or nearly empty."""
    idx, p = W.random_cells(n, count, radius, seed=7 + n)
    ref = _run(n, prec, gbees.GBEES_LAUNCH_GRAPH, 0, idx, p, 3)
    for blocks in (1, 3, 0):
        got = _run(n, prec, gbees.GBEES_LAUNCH_PERSISTENT, blocks, idx, p, 3)
        assert got[4] == ref[4]
        for x, y in zip(got[:4], ref[:4]):
            assert np.array_equal(x, y)
