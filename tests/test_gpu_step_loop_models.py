"""The step loop of a small grid against the kernels of a large one, in every drift model
and at the edge of the key range. The drift models are written twice on the device (by
cell, and by face for the new cells of the step loop) and have to agree to the last bit."""
import numpy as np
import pytest

from paper_2508_13986_gb300 import gbees
from paper_2508_13986_gb300 import workloads as W

pytestmark = pytest.mark.gpu

PREC = pytest.mark.parametrize("prec", [gbees.GBEES_FP64, gbees.GBEES_FP32])
MODES = (gbees.GBEES_LAUNCH_GRAPH, gbees.GBEES_LAUNCH_DIRECT, gbees.GBEES_LAUNCH_PERSISTENT)


@PREC
@pytest.mark.parametrize("n,dyn,params", [
    (1, gbees.GBEES_DYN_CONSTANT, [-0.7]), (4, gbees.GBEES_DYN_CONSTANT, [0.7, -0.3, 0.0, 1.1]),
    (2, gbees.GBEES_DYN_LINEAR, [0.1, -1.3, 0.9, -0.2, 0.05, -0.4]),
    (3, gbees.GBEES_DYN_LORENZ63, [10.0, 28.0, 8.0 / 3.0]),
    (3, gbees.GBEES_DYN_LORENZ63_SHIFTED, [4.0, 1.0, 48.0]),
    (4, gbees.GBEES_DYN_LORENZ96, [4.0]), (5, gbees.GBEES_DYN_LORENZ96, [8.1]), (6, gbees.GBEES_DYN_LORENZ96, [4.0])])
def test_both_forms_of_a_drift_model_agree(n, dyn, params, prec):
    """Random cells (a new cell for nearly every old one), widths that are no powers of
    two, three prunes: the same bits from every launch mode."""
    idx, p = W.random_cells(n, {1: 200, 2: 3000}.get(n, 2500), {1: 150, 2: 40, 3: 12, 4: 6}.get(n, 4), seed=21 + n)
    h = np.array([0.3, 0.7, 0.45, 0.6, 0.35, 0.55])[:n]
    x0 = np.array([-1.3, 2.1, 9.7, -0.4, 3.3, 0.9])[:n]
    speed = {gbees.GBEES_DYN_LORENZ63: 4e-3, gbees.GBEES_DYN_LORENZ63_SHIFTED: 4e-3}.get(dyn, 4e-2)
    runs = []
    for mode in MODES:
        cfg = gbees.make_config(n, dyn, params, h, x0, 1e-3, 0.9, 2, prec, max_cells=1 << 22, launch_mode=mode)
        g = gbees.Grid(cfg)
        g.init_cells(idx, p)
        st = [g.propagate(t) for t in (0.5 * speed, speed)]
        runs.append((*g.read_cells(), *g.moments(), [(s.steps, s.cell_updates, s.n_cells, s.t, s.norm) for s in st]))
        g.close()
    for got in runs[1:]:
        assert got[4] == runs[0][4]
        for x, y in zip(got[:4], runs[0][:4]):
            assert np.array_equal(x, y)


@PREC
@pytest.mark.parametrize("n", [1, 3, 6])
@pytest.mark.parametrize("side", [-1, 1])
def test_growth_to_the_end_of_the_key_range(n, side, prec):
    """A cell carried towards the last index that has a key: the same densities on the
    way, then GBEES_EKEYRANGE, in every launch mode."""
    top = 2 ** ((32 if n == 1 else 63 // n) - 1) - 1
    idx = np.zeros((1, n), dtype=np.int32)
    idx[0, 0] = side * (top - 6)
    drift = [0.0] * n
    drift[0] = float(side)
    runs = []
    for mode in MODES:
        cfg = gbees.make_config(n, gbees.GBEES_DYN_CONSTANT, drift, [0.5] * n, [0.0] * n, 1e-3, 0.9, 20, prec,
                                max_cells=1 << 14, launch_mode=mode)
        g = gbees.Grid(cfg)
        g.init_cells(idx, np.ones(1))
        st = g.propagate(0.9)
        runs.append((*g.read_cells(), (st.steps, st.n_cells, st.t)))
        with pytest.raises(gbees.GbeesError) as e:
            g.propagate(20.0)
        assert e.value.status == gbees.GBEES_EKEYRANGE
        g.close()
    for got in runs[1:]:
        assert got[2] == runs[0][2] and np.array_equal(got[0], runs[0][0]) and np.array_equal(got[1], runs[0][1])
