"""The workspace holds every array that the kernels address, the update's pairs (two
values per entry and dimension in one block) among them: its size is the sum of the
arrays, each on a 256-byte boundary, at odd and even capacities."""
import pytest

from paper_2508_13986_gb300 import gbees


def _up(x):
    return (x + 255) // 256 * 256


@pytest.mark.parametrize("prec,S", [(gbees.GBEES_FP64, 8), (gbees.GBEES_FP32, 4)])
@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 6])
def test_workspace_holds_every_array(n, prec, S):
    for cap in (1, 2, 31, 63, 64, 1000, 4097, 65535):
        cfg = gbees.make_config(n, gbees.GBEES_DYN_CONSTANT, [0.0] * n, [1.0] * n, [0.0] * n, precision=prec,
                                max_cells=cap)
        slots = 64
        while slots < 2 * cap:
            slots *= 2
        rows = S * n * cap
        per_generation = [8 * cap, S * cap, 8 * n * cap, 2 * cap, 4 * cap, rows, 8 * cap]
        total = sum(2 * _up(b) for b in per_generation)
        total += _up(2304) + _up(16 * 8193) + _up(64 * 8192) + _up(4 * 256 * 1024)   # scalars, counts, partials, digits
        total += _up(cap) + _up(4 * cap) + _up(16 * slots)                           # keep, map, table
        pairs = _up(rows) + _up(rows)
        assert pairs >= 2 * rows
        total += pairs + _up(S * cap) + _up(rows)                                    # pairs, tg, fluxes
        assert gbees.gbees_workspace_bytes(cfg) == total, (n, cap)
