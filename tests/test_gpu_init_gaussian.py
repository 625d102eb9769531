"""The initial Gaussian against the oracle: the same set of cells and the same
densities, whatever the scale, the origin and the shape of the prior.

The library sweeps the box by rows in single precision and decides the cells near
the limit in FP64; the oracle evaluates every cell of the box in FP64."""
import numpy as np
import pytest

from oracle.oracle import DYN_CONSTANT, LIM_MC, Oracle
from paper_2508_13986_gb300 import gbees

pytestmark = pytest.mark.gpu

THR = 1e-6


def _cov(n, sigma, corr):
    """Covariance with standard deviations sigma, its correlations products of
    components of a vector (the largest is corr)."""
    a = np.sqrt(corr) * np.array([1.0, -0.9, 0.8, 0.95, -0.7, 0.6])[:n]
    C = np.outer(a, a)
    np.fill_diagonal(C, 1.0)
    return C * np.outer(sigma, sigma)


def _check(n, sigma, per, origin, shift, corr, prec, thr=THR):
    """per: cells per standard deviation; origin: x0 in standard deviations;
    shift: the mean's distance from x0 in cells."""
    sigma = np.asarray(sigma, dtype=np.float64)
    h = sigma / np.asarray(per, dtype=np.float64)
    x0 = np.asarray(origin, dtype=np.float64) * sigma
    mean = x0 + np.asarray(shift, dtype=np.float64) * h
    cov = _cov(n, sigma, corr)
    drift = [0.0] * n
    o = Oracle(n, DYN_CONSTANT, drift, list(h), list(x0), thr, 0.9, 20, LIM_MC)
    o.init_gaussian(mean, cov)
    cfg = gbees.make_config(n, gbees.GBEES_DYN_CONSTANT, drift, h, x0, thr, precision=prec, max_cells=1 << 22)
    g = gbees.Grid(cfg)
    g.init_gaussian(mean, cov)
    gi, gp = g.read_cells()
    g.close()
    oi, op = o.read_cells()
    assert gi.shape == oi.shape and np.array_equal(gi, oi), (gi.shape, oi.shape)
    # the two inverses of cov differ by a few roundings times its condition (below 20),
    # the exponents (up to 14) by as much: 14 * 20 * 36 * 2^-53 < 2e-12; FP32 storage
    # rounds a density and their sum by 2^-24 each
    tol = 2e-12 * max(1.0, -np.log(thr) / 14.0)  # (a smaller threshold: larger exponents)
    if prec == gbees.GBEES_FP32:
        tol += 2.5 * 2.0 ** -24
    assert np.max(np.abs(gp / op - 1.0)) <= tol


PREC = pytest.mark.parametrize("prec", [gbees.GBEES_FP64, gbees.GBEES_FP32])


@PREC
@pytest.mark.parametrize("n,per", [(1, 50.0), (2, 9.0), (3, 5.0), (4, 2.0), (5, 1.5), (6, 1.2)])
@pytest.mark.parametrize("corr", [0.0, 0.5])
def test_shifted_and_correlated_priors(n, per, corr, prec):
    _check(n, np.linspace(0.3, 2.0, n), per, np.linspace(-3.0, 4.0, n), np.linspace(0.37, -4.4, n), corr, prec)


@PREC
@pytest.mark.parametrize("corr", [0.0, 0.5])
@pytest.mark.parametrize("sigma", [(1e21,) * 3, (1e22,) * 3, (1e23,) * 3, (1e22, 1e4, 1e4), (1e4, 1e4, 1e22),
                                   (1e30, 1e-30, 1.0), (1e-25,) * 3, (1e60,) * 3])
def test_any_scale(sigma, corr, prec):
    _check(3, sigma, 4.0, [0.0, 1.0, -2.0], [0.0, 0.3, -0.4], corr, prec)


@PREC
@pytest.mark.parametrize("corr", [0.0, 0.5])
@pytest.mark.parametrize("origin", [1e12, -1e13, 1e14, 1e15])
def test_an_origin_far_from_zero(origin, corr, prec):
    """The centres x0 + i h are spaced by roundings of x0 there (2^-53 origin is up
    to an eighth of a standard deviation)."""
    _check(3, [0.7, 1.0, 1.3], 4.0, [origin] * 3, [0.0, 3.0, -2.0], corr, prec)


@PREC
@pytest.mark.parametrize("per", [(140.0, 1.0, 1.0), (0.6, 100.0, 30.0), (1.0, 1.0, 97.1), (1.0, 1.0, 150.0)])
def test_long_axes_and_rows(per, prec):
    """Axes beyond the table of 1024 distances, rows around and beyond 1024 cells."""
    _check(3, [1.0, 1.0, 1.0], per, [0.0, 0.5, 0.0], [0.2, 0.0, -0.3], 0.3, prec)


@PREC
@pytest.mark.parametrize("thr,per", [(1e-285, 0.7), (1e-295, 0.7), (1e-290, 0.4)])
def test_tiny_thresholds(thr, per, prec):
    """Thresholds around the one below which FP64 decides on every cell (FP32 stores 0
    below 1e-45)."""
    _check(3, [1.0, 0.8, 1.2], per, [0.0, 0.5, -1.0], [0.1, -0.2, 0.0], 0.3, prec,
           thr if prec == gbees.GBEES_FP64 else 1e-30)
