"""The initial Gaussian's rows in single precision (csrc/gbees_rows.cuh), built for the
host: what they decide is what FP64 decides, at any scale, origin and shape of the
prior; what they leave to FP64 is little where the prior is ordinary."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2508_13986_gb300", "csrc")
SRC = r"""
#include "gbees_rows.cuh"
using namespace gbees;
template <int N>
static void rows_of(const float* dx, long rows, const float* w, int len, float slack, float qlim, signed char* side) {
    for (long r = 0; r < rows; ++r) {
        const InitRow f = row_form<N>(dx + r * N, w, (float)len, slack);
        for (int i = 0; i < len; ++i) {
            float e;
            const float d = row_gap(f, i, qlim, e);
            side[r * len + i] = d > e ? 1 : d < -e ? -1 : 0;  // out, in, left to FP64
        }
    }
}
extern "C" void sides(int n, const float* dx, long rows, const float* w, int len, float slack, float qlim,
                      signed char* side) {
    if (n == 3) rows_of<3>(dx, rows, w, len, slack, qlim, side);
    if (n == 4) rows_of<4>(dx, rows, w, len, slack, qlim, side);
    if (n == 5) rows_of<5>(dx, rows, w, len, slack, qlim, side);
    if (n == 6) rows_of<6>(dx, rows, w, len, slack, qlim, side);
}
extern "C" double slack_of(double x0, double h, double i) { return centre_slack(x0, h, i); }
extern "C" double above(int n, const double* icov, const double* h, const double* dx, const double* s) {
    return form_above(n, icov, h, dx, s);
}
"""
P, D, F = ctypes.c_void_p, ctypes.c_double, ctypes.c_float
THR = 1e-6


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("rows")
    src, so = d / "r.cpp", d / "r.so"
    src.write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, str(src), "-o",
                    str(so)], check=True)
    L = ctypes.CDLL(str(so))
    L.sides.argtypes = [ctypes.c_int, P, ctypes.c_long, P, ctypes.c_int, F, F, P]
    L.slack_of.restype = L.above.restype = D
    L.slack_of.argtypes = [D, D, D]
    L.above.argtypes = [ctypes.c_int, P, P, P, P]
    return L


def _prior(n, sigma, corr, g):
    a = np.sqrt(corr) * g.uniform(-1.0, 1.0, n)
    C = np.outer(a, a)
    np.fill_diagonal(C, 1.0)
    # the inverse scaled from that of the correlations (no overflow on the way)
    return np.linalg.inv(C) / np.outer(sigma, sigma)


def _sides(lib, n, sigma, per, origin, corr, seed, thr=THR, rows=1500, qlim=None):
    """(side of every cell of some rows, whether FP64 puts it in the set, FP64's q)."""
    g = np.random.Generator(np.random.PCG64(seed))
    sigma = np.broadcast_to(np.asarray(sigma, dtype=np.float64), n)
    h = sigma / per
    x0 = origin * sigma
    mean = x0 + g.uniform(-3.0, 3.0, n) * h
    icov = _prior(n, sigma, corr, g)
    limit = -2.0 * np.log(thr)
    ctr = np.round((mean - x0) / h)
    hw = np.ceil(np.sqrt(limit) * sigma / h) + 1.0
    idx = ctr + np.round(g.uniform(-1.0, 1.0, (rows, n)) * hw)
    idx[: rows // 2] = ctr + np.round(g.uniform(-0.4, 0.4, (rows // 2, n)) * hw)
    idx[:, -1] = ctr[-1] - hw[-1]
    length = int(2 * hw[-1] + 1)
    with np.errstate(over="ignore", invalid="ignore"):
        dx = (((x0 + idx * h) - mean) * (1.0 / h)).astype(np.float32)
        w = (icov * h[:, None] * h[None, :]).astype(np.float32)
    slack = lib.slack_of(x0[-1], h[-1], abs(ctr[-1]) + hw[-1] + 1)
    side = np.zeros((rows, length), dtype=np.int8)
    lib.sides(n, dx.ctypes.data, rows, w.ctypes.data, length, slack, limit if qlim is None else qlim, side.ctypes.data)
    cells = np.repeat(idx[:, None, :], length, axis=1)
    cells[:, :, -1] += np.arange(length)
    d = (x0 + cells * h) - mean
    with np.errstate(over="ignore", invalid="ignore"):
        q = sum((d[..., a] * icov[a, c]) * d[..., c] for a in range(n) for c in range(n))
    return side, np.exp(-0.5 * q) > thr, q


@pytest.mark.parametrize("corr", [0.0, 0.6])
@pytest.mark.parametrize("n,per", [(3, 4.0), (3, 60.0), (4, 3.0), (5, 2.0), (6, 1.3), (6, 0.4)])
@pytest.mark.parametrize("scale", [1.0, 1e-30, 1e-15, 1e15, 1e19, 1e22, 1e40, 1e100])
def test_rows_decide_as_fp64_at_any_scale(lib, n, per, scale, corr):
    side, inside, _ = _sides(lib, n, scale, per, 2.0, corr, n)
    assert not np.any(side[inside] > 0) and not np.any(side[~inside] < 0)
    assert inside.any() and (~inside).any() and np.mean(side == 0) < 0.01


@pytest.mark.parametrize("corr", [0.0, 0.6])
@pytest.mark.parametrize("scales", [(1e22, 1e4, 1e4), (1e4, 1e4, 1e22), (1e30, 1e-30, 1.0), (1e-40, 1e40, 1e-10)])
def test_rows_decide_as_fp64_at_mixed_scales(lib, scales, corr):
    side, inside, _ = _sides(lib, 3, scales, 5.0, -1.0, corr, 9)
    assert not np.any(side[inside] > 0) and not np.any(side[~inside] < 0)
    assert np.mean(side == 0) < 0.01


@pytest.mark.parametrize("corr", [0.0, 0.6])
@pytest.mark.parametrize("origin", [1e6, -1e10, 1e12, 1e13, -1e14, 1e15, 1e16])
@pytest.mark.parametrize("n,per", [(3, 4.0), (3, 40.0), (5, 2.0)])
def test_rows_decide_as_fp64_far_from_zero(lib, n, per, origin, corr):
    for seed in range(4):
        side, inside, _ = _sides(lib, n, np.linspace(0.7, 1.3, n), per, origin, corr, seed)
        assert not np.any(side[inside] > 0) and not np.any(side[~inside] < 0)


@pytest.mark.parametrize("per", [1e-3, 1e-12, 1e-30, 1e-160])
def test_cells_far_wider_than_the_prior_are_decided_or_left_to_fp64(lib, per):
    side, inside, _ = _sides(lib, 3, 1.0, per, 0.0, 0.3, 4)
    assert not np.any(side[inside] > 0) and not np.any(side[~inside] < 0)


def test_an_infinite_limit_leaves_every_cell_to_fp64(lib):
    side, _, _ = _sides(lib, 4, 1.0, 2.0, 1.0, 0.4, 3, qlim=np.inf)
    assert not side.any()


@pytest.mark.parametrize("origin", [0.0, 1e13, 1e15])
@pytest.mark.parametrize("scale", [1.0, 1e22])
def test_the_first_pass_keeps_the_cell_with_the_largest_density(lib, origin, scale):
    """Limit: the form at the cell nearest the mean, from above (form_above)."""
    for seed in range(20):
        g = np.random.Generator(np.random.PCG64(seed))
        sigma = scale * np.array([0.7, 1.0, 1.3])
        h, x0 = sigma / 2.0, origin * sigma
        mean = x0 + g.uniform(-3.0, 3.0, 3) * h
        icov = _prior(3, sigma, 0.9, g)
        ctr = np.round((mean - x0) / h)
        near = np.array([lib.slack_of(x0[k], h[k], abs(ctr[k]) + 13) for k in range(3)])
        dx = ((x0 + ctr * h) - mean) / h
        qlim = lib.above(3, icov.ctypes.data, h.ctypes.data, dx.ctypes.data, near.ctypes.data)
        i = np.arange(-12, 13)
        rows = np.stack(np.meshgrid(i, i, [-12], indexing="ij"), axis=-1).reshape(-1, 3) + ctr
        f = (((x0 + rows * h) - mean) * (1.0 / h)).astype(np.float32)
        w = (icov * h[:, None] * h[None, :]).astype(np.float32)
        side = np.zeros((rows.shape[0], 25), dtype=np.int8)
        lib.sides(3, f.ctypes.data, rows.shape[0], w.ctypes.data, 25, near[2], qlim, side.ctypes.data)
        cells = np.repeat(rows[:, None, :], 25, axis=1)
        cells[:, :, -1] += np.arange(25)
        d = (x0 + cells * h) - mean
        q = sum((d[..., a] * icov[a, c]) * d[..., c] for a in range(3) for c in range(3))
        best = np.unravel_index(np.argmin(q), q.shape)
        assert side[best] <= 0
