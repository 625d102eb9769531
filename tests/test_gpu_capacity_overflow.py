"""A pool that outgrows its capacity by far in one step answers GBEES_ECAPACITY soon: the
claims that go on until the phase ends do not search a full table slot by slot (on one
block they did, for minutes)."""
import time

import numpy as np
import pytest

from paper_2508_13986_gb300 import gbees
from paper_2508_13986_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [gbees.GBEES_FP64, gbees.GBEES_FP32])
@pytest.mark.parametrize("blocks", [1, 0])
@pytest.mark.parametrize("cap", [4096, 1 << 16])
def test_an_overflowing_pool_answers_soon(cap, blocks, prec):
    idx, p = W.random_cells(6, 300, 12, seed=4)  # (scattered cells: twelve halo cells and 15 edges each)
    cfg = gbees.make_config(6, gbees.GBEES_DYN_LORENZ96, [4.0], [0.5] * 6, [1.0] * 6, 1e-9, 0.9, 3, prec, max_cells=cap,
                            launch_mode=gbees.GBEES_LAUNCH_PERSISTENT)
    g = gbees.Grid(cfg)
    assert gbees.gbees_set_persist_blocks(g.ctx, blocks) == gbees.GBEES_OK
    t0 = time.perf_counter()
    with pytest.raises(gbees.GbeesError) as e:
        g.init_cells(idx, p)
        g.propagate(1.0)
    assert e.value.status == gbees.GBEES_ECAPACITY
    assert time.perf_counter() - t0 < 10.0
    small = gbees.make_config(6, gbees.GBEES_DYN_LORENZ96, [4.0], [0.5] * 6, [1.0] * 6, 1e-9, 0.9, 3, prec,
                              max_cells=1 << 16, launch_mode=gbees.GBEES_LAUNCH_PERSISTENT)
    h = gbees.Grid(small)
    for k in range(2):  # a batch in queue mode, one block per grid; usable again after it
        h.init_cells(idx[:20], p[:20])
        t0 = time.perf_counter()
        with pytest.raises(gbees.GbeesError) as e:
            gbees.propagate_batch([h], [1.0], 0, 1)
        assert e.value.status == gbees.GBEES_ECAPACITY
        assert time.perf_counter() - t0 < 10.0
    g.close()
    h.close()
