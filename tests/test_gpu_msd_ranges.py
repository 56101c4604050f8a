"""lb_msd_trajectory on trajectories whose columns range over far more than the
displacements that a lag averages: a record far away, a loop that comes back,
drift from rest, values about 0. Against numpy in extended precision.

Tolerance: an FP64 evaluation rounds each squared difference by up to 2^-52
relative (difference and square) and a sum of n terms by as much again per
level of its tree, log2(n) + 8 levels at most: (log2 n + 10) 2^-52 relative
to the average itself, for every lag."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _still(n):
    q = np.zeros((n, 4))
    q[:, 0] = 1.0
    return q


def _check(X, lags):
    from paper_1604_01829_gb300 import lb
    got = lb.lb_msd_trajectory(X, _still(len(X)), lags)[0, :, :3]
    L = X.astype(np.longdouble)
    ref = np.stack([((L[l:] - L[:-l]) ** 2).mean(axis=0) for l in range(1, lags + 1)])
    n = len(X) - np.arange(1, lags + 1)
    assert np.all(np.abs(got - ref) <= (np.log2(n) + 10)[:, None] * 2.0 ** -52 * ref)


@pytest.mark.parametrize("far", [1e2, 1e6, 1e12])
@pytest.mark.parametrize("nrec,at", [(9, 4), (200, 100), (200, 90), (1000, 540)])
def test_one_record_far_away(nrec, at, far):
    rng = np.random.default_rng(nrec + at)
    X = 0.05 * rng.standard_normal((nrec, 3))
    X[at, 0] += far
    X[at, 1] -= far
    _check(X, nrec - 1)


def test_a_loop_that_comes_back():
    t = np.arange(400)
    X = np.stack([1e3 * np.sin(2 * np.pi * t / 399), 1e-3 * t, 5.0 * np.cos(2 * np.pi * t / 399)], axis=1)
    X += 1e-6 * np.random.default_rng(2).standard_normal(X.shape)
    _check(X, 399)


def test_drift_from_rest_and_values_about_zero():
    rng = np.random.default_rng(3)
    t = np.arange(700.0)
    X = np.stack([0.01 * t * t, np.cumsum(0.05 * rng.standard_normal(700)), 1e-9 * rng.standard_normal(700)], axis=1)
    _check(X, 699)
