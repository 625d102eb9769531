"""A drift that is no number in one component. In FP64 the step ends with
GBEES_EDEGENERATE; in FP32 a face whose velocity is no number carries no flux, and the
call returns the density with its mass, in every launch mode alike."""
import numpy as np
import pytest

from paper_2508_13986_gb300 import gbees
from paper_2508_13986_gb300 import workloads as W

pytestmark = pytest.mark.gpu

MODES = (gbees.GBEES_LAUNCH_PERSISTENT, gbees.GBEES_LAUNCH_GRAPH, gbees.GBEES_LAUNCH_DIRECT)


def _run(n, prec, mode):
    idx, p = W.random_cells(n, 200, 8, seed=2)
    drift = [0.3] * n
    drift[0] = float("nan")
    cfg = gbees.make_config(n, gbees.GBEES_DYN_CONSTANT, drift, [0.5] * n, [0.1] * n, 1e-3, 0.9, 3, prec,
                            max_cells=1 << 18, launch_mode=mode)
    g = gbees.Grid(cfg)
    g.init_cells(idx, p / (0.5 ** n * p.sum()))
    s = g.propagate(0.2)
    return (*g.read_cells(), s)


@pytest.mark.parametrize("n", [2, 4])
def test_fp32_leaves_out_what_is_no_number(n):
    runs = [_run(n, gbees.GBEES_FP32, m) for m in MODES]
    i, p, s = runs[0]
    assert np.all(np.isfinite(p)) and abs(s.norm - 1.0) < 1e-5  # (exact sums of values rounded to 2^-24)
    for j, q, z in runs[1:]:
        assert np.array_equal(i, j) and np.array_equal(p, q) and z == s


@pytest.mark.parametrize("mode", MODES)
def test_fp64_ends_with_a_status(mode):
    with pytest.raises(gbees.GbeesError) as e:
        _run(3, gbees.GBEES_FP64, mode)
    assert e.value.status == gbees.GBEES_EDEGENERATE
