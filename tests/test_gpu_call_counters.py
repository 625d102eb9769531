"""The counters of the last propagate call, after calls that read the scalars back."""
import numpy as np
import pytest

from paper_2508_13986_gb300 import gbees
from paper_2508_13986_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [gbees.GBEES_LAUNCH_PERSISTENT, gbees.GBEES_LAUNCH_GRAPH, gbees.GBEES_LAUNCH_DIRECT])
def test_a_propagate_without_steps_leaves_zero_counters(mode):
    w = W.lorenz63(h=0.25, t_end=0.02)  # (a pool above the rank read-out's 2^14 entries)
    g = gbees.grid_for_workload(w, max_cells=1 << 18, launch_mode=mode)
    g.init_gaussian(w.mean, w.cov)
    first = g.propagate(w.t_end)
    assert first.steps > 0 and first.cell_updates > 0 and first.n_pool > 1 << 14
    for t in (w.t_end, 0.5 * w.t_end):
        again = g.propagate(t)
        assert (again.steps, again.cell_updates) == (0, 0)
        for read in (g.moments, g.read_cells, lambda: g.correct_gaussian([-11.0], np.eye(1), [0])):
            read()
            s = g.stats()
            assert (s.steps, s.cell_updates) == (0, 0)
            assert s.t == first.t and s.total_steps == first.steps
    g.close()
