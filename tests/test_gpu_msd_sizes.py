"""lb_msd_trajectory at the edges of its tiles (15 origins a lane, 480 a
tile, 3840 between two sums, 8 or 4 lags a warp, 64 or 32 a block), at angles
beyond 90 degrees, with far offsets, at rest, and with a value that is not
finite, against the plain FP64 averages.

Tolerances: the differences are exact to 2^-57 of a column's range and the
squares are summed exactly, so the averages of the columns agree to the
rounding of the reference, 1e-12 relative to the column's largest value
covers the sums of up to 5000 terms; the angle's polynomial is good to 2^-55
and its inputs (unit vectors to 2^-53) to 1e-16 / theta, theta > 1e-3 here."""
import numpy as np
import pytest

from perf import cases

pytestmark = pytest.mark.gpu


def _walk(nb, nrec, seed, turn=0.05, step=0.05, at=30.0):
    from paper_1604_01829_gb300 import workloads as W
    rng = np.random.default_rng(seed)
    X = at + np.cumsum(step * rng.standard_normal((nb, nrec, 3)), axis=1)
    q = np.zeros((nb, nrec, 4))
    for b in range(nb):
        cur = W.random_unit_quaternion(rng)
        for k in range(nrec):
            h = 0.5 * turn * rng.standard_normal(3)
            d = np.concatenate([[np.sqrt(max(0.0, 1 - h @ h))], h])
            w0, v0, w1, v1 = cur[0], cur[1:], d[0], d[1:]
            cur = np.concatenate([[w0 * w1 - v0 @ v1], w0 * v1 + w1 * v0 + np.cross(v0, v1)])
            cur /= np.linalg.norm(cur)
            q[b, k] = cur
    return X, q


def _check(X, q, lags):
    import torch
    from paper_1604_01829_gb300 import lb
    got = lb.lb_msd_trajectory(X, q, lags)
    orig = cases._trajectories
    cases._trajectories = lambda c, seed: (X, q)
    try:
        with torch.no_grad():
            ref = cases._exact_msd(dict(lags=lags), 0)["msd"].cpu().numpy()
    finally:
        cases._trajectories = orig
    scale = np.abs(ref).max(axis=1, keepdims=True)
    assert np.all(np.abs(got - ref) <= 1e-12 * scale + 1e-300)


@pytest.mark.parametrize("nrec,lags", [(2, 1), (3, 2), (16, 15), (33, 9), (480, 479), (481, 64), (489, 65), (545, 33),
                                       (961, 128), (3900, 40), (4400, 17)])
def test_sizes(nrec, lags):
    _check(*_walk(2, nrec, nrec), lags)


def test_angles_beyond_a_right_angle():
    _check(*_walk(3, 300, 5, turn=1.2), 250)


def test_far_offset_and_position_at_rest():
    X, q = _walk(3, 200, 6, at=1e6, step=1e-3)
    X[2] = X[2, :1]
    X[1, :, 2] = np.linspace(-1e4, 1e4, 200)
    _check(X, q, 60)


def test_values_that_are_not_finite_reach_their_lags_only():
    from paper_1604_01829_gb300 import lb
    X, q = _walk(2, 40, 7)
    clean = lb.lb_msd_trajectory(X, q, 35)
    X[0, 20, 1] = np.nan
    got = lb.lb_msd_trajectory(X, q, 35)
    assert np.array_equal(got[1], clean[1])
    hit = np.array([any(t == 20 or t + l == 20 for t in range(40 - l)) for l in range(1, 36)])
    assert np.array_equal(np.isnan(got[0, :, 1]), hit)
    fine = [0, 2, 6, 7, 8, 9]
    assert np.allclose(got[0][:, fine], clean[0][:, fine], rtol=1e-12, atol=1e-300)
