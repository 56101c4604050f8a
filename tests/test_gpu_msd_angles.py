"""The squared angle of lb_msd_trajectory (column 6) between reference vectors
that stand at a chosen angle: records alternate between two orientations a
rotation apart, so that every odd lag's average is that one pair's value.

The expected value is the angle of the rotation itself, about the x axis with
the reference vector along z. Tolerance: the vectors come from quaternions and
rotation matrices rounded in FP64 (an angle error of up to 4e-16 each) and
the evaluation is good to 2^-52 relative: 2 theta (8e-16) + 2e-16 theta^2
< 6e-15 for theta up to pi."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOL = 6e-15


def _squared_angles(qa, qb, lags=5, nrec=64):
    from paper_1604_01829_gb300 import lb
    q = np.zeros((1, nrec, 4))
    q[0, 0::2], q[0, 1::2] = qa, qb
    return lb.lb_msd_trajectory(np.zeros((1, nrec, 3)) + 1.0, q, lags, p_ref=(0, 0, 1))[0, :, 6]


def _about_x(angle):
    return [np.cos(angle / 2), np.sin(angle / 2), 0.0, 0.0]


@pytest.mark.parametrize("qb", [(0.5, 0.5, 0.5, 0.5), (np.sqrt(0.5), np.sqrt(0.5), 0, 0), (np.sqrt(0.5), 0, -np.sqrt(0.5), 0)])
def test_quarter_turns(qb):
    got = _squared_angles((1, 0, 0, 0), qb)
    assert np.abs(got[0::2] - np.pi ** 2 / 4).max() <= TOL
    assert np.abs(got[1::2]).max() <= TOL


@pytest.mark.parametrize("off", [1e-16, 1e-13, 1e-12, 1e-11, 1e-10, 2e-10, 2.4e-10, 3e-10, 1e-9, 1e-6])
@pytest.mark.parametrize("side", [-1, 1])
def test_angles_close_to_a_right_angle(off, side):
    angle = np.pi / 2 + side * off
    got = _squared_angles((1, 0, 0, 0), _about_x(angle))
    assert np.abs(got[0::2] - angle ** 2).max() <= TOL
    assert np.abs(got[1::2]).max() <= TOL


def test_random_perpendicular_pairs():
    """Pairs of rotations whose reference vectors are perpendicular to rounding, in any direction."""
    from paper_1604_01829_gb300 import lb
    rng = np.random.default_rng(4)
    nb = 400
    q = np.zeros((nb, 2, 4))
    for b in range(nb):
        p, r = rng.standard_normal((2, 3))
        p /= np.linalg.norm(p)
        r -= p * (p @ r)
        r /= np.linalg.norm(r)
        for k, v in enumerate((p, r)):                    # the rotation that takes z to v
            h = np.array([1.0 + v[2], -v[1], v[0], 0.0])
            q[b, k] = h / np.linalg.norm(h)
    got = lb.lb_msd_trajectory(np.zeros((nb, 2, 3)), q, 1, p_ref=(0, 0, 1))[:, 0, 6]
    # the frames built above are perpendicular to a few roundings, more for p or r close to -z
    assert np.abs(got - np.pi ** 2 / 4).max() <= 1e-12


def test_angles_beyond_a_right_angle_are_not_biased():
    """Supplements s from 0.07 rad to a right angle, thousands of pairs each,
    beside an extended-precision evaluation from the same quaternions
    (arctangent of cross and dot product): the sum of the vectors is held to
    1/2 unit of 2^-54 squared, an error of 2^-55 / s per pair in theta and no
    bias, so the average of n pairs stays within theta 2^-54 / s / sqrt(n) of
    the exact value; 2 units of 2^-52 cover the rounding of the result."""
    from paper_1604_01829_gb300 import lb
    rng = np.random.default_rng(9)
    nrec = 4000
    for s in (0.07, 0.1, 0.2, 0.5, 1.0, 1.5):
        q = np.zeros((1, nrec, 4))
        # alternating records: turned about a common random axis by 0 and pi - s, each with its own small jitter
        q[0, :, 0] = 1.0
        q[0, 1::2] = _about_x(np.pi - s)
        q[0] += 1e-3 * s * rng.standard_normal((nrec, 4))
        q /= np.linalg.norm(q, axis=2, keepdims=True)
        got = lb.lb_msd_trajectory(np.zeros((1, nrec, 3)), q, 1, p_ref=(0, 0, 1))[0, 0, 6]
        w, x, y, z = q[0].astype(np.longdouble).T
        p = np.stack([2 * (x * z + y * w), 2 * (y * z - x * w), 1 - 2 * (x * x + y * y)], axis=1)
        a, b = p[:-1], p[1:]
        cr = np.stack([a[:, 1] * b[:, 2] - a[:, 2] * b[:, 1], a[:, 2] * b[:, 0] - a[:, 0] * b[:, 2],
                       a[:, 0] * b[:, 1] - a[:, 1] * b[:, 0]], axis=1)
        th = np.arctan2(np.sqrt((cr * cr).sum(1)), (a * b).sum(1))
        ref = float((th * th).mean())
        assert abs(got - ref) <= 2 * 2.0 ** -52 * ref


@pytest.mark.parametrize("side", [1 - 1e-9, 1.0, 1 + 1e-9])
@pytest.mark.parametrize("power", range(-10, 2))
def test_supplements_at_every_scaling_switch(power, side):
    """Squared chords of the supplement on both sides of each power of two,
    where the square root's argument is scaled anew (below 2^-8: FP64). Half a
    unit of 2^-54 in the chord's square is 2^-55 / s in theta."""
    s = 2 * np.arcsin(0.5 * np.sqrt(side * 2.0 ** power))
    got = _squared_angles((1, 0, 0, 0), _about_x(np.pi - s))
    assert np.abs(got[0::2] - (np.pi - s) ** 2).max() <= TOL + 2 * np.pi * 2.0 ** -55 / s


@pytest.mark.parametrize("qb", [(0, 0.5, 0.5, 0), (0, 0.5 * (1 - 2.0 ** -40), 0.5, 0), (0, 3e100, 1e90, 0)])
def test_quaternions_that_leave_no_unit_vector(qb):
    """Quaternions far from unit length whose matrix takes the reference vector
    to 0, nearly to 0 or beyond the squares' range: the angle is the
    arctangent's of the vectors as they are (0 between a vector and 0)."""
    w, x, y, z = qb
    p = np.array([2 * (x * z + y * w), 2 * (y * z - x * w), 1 - 2 * (x * x + y * y)])
    with np.errstate(over="ignore", invalid="ignore"):
        th = np.arctan2(np.hypot(p[0], p[1]), p[2])        # against (0, 0, 1)
    got = _squared_angles((1, 0, 0, 0), qb)
    assert np.abs(got[0::2] - th ** 2).max() <= TOL
    assert np.abs(got[1::2]).max() <= TOL


@pytest.mark.parametrize("nb,nrec,lags", [(1, 481, 1), (1, 482, 9), (1, 4000, 5), (1, 4400, 400), (3, 1700, 33), (2, 3900, 3899), (40, 600, 64), (20, 4000, 20)])
def test_few_bodies_and_lags(nb, nrec, lags):
    """Tiles split over blocks, one or four lags a warp: small and large angles
    together, against FP64's own evaluation. Its arctangents and unit vectors are
    good to 4e-16 + 2^-52 relative, sums of n terms to (log2 n + 8) 2^-52."""
    from paper_1604_01829_gb300 import lb
    rng = np.random.default_rng(nrec + lags)
    q = np.zeros((nb, nrec, 4))
    q[..., 0] = 1.0
    q[:, 1:, 1:] = np.cumsum(0.3 * rng.standard_normal((nb, nrec - 1, 3)), axis=1)
    q /= np.linalg.norm(q, axis=2, keepdims=True)
    got = lb.lb_msd_trajectory(np.zeros((nb, nrec, 3)), q, lags, p_ref=(0, 0, 1))[:, :, 6]
    w, x, y, z = np.moveaxis(q, 2, 0)
    p = np.stack([2 * (x * z + y * w), 2 * (y * z - x * w), 1 - 2 * (x * x + y * y)], axis=2)
    for l in {1, 2, lags // 2 + 1, max(1, lags - 1), lags}:
        if l > lags:
            continue
        a, b = p[:, :-l], p[:, l:]
        th = np.arctan2(np.linalg.norm(np.cross(a, b), axis=2), (a * b).sum(2))
        n = nrec - l
        ref = (th * th).mean(axis=1)
        bound = 2 * th.mean(axis=1) * 4e-16 + (np.log2(n) + 10) * 2.0 ** -52 * ref
        assert np.all(np.abs(got[:, l - 1] - ref) <= bound + 4 * np.finfo(float).eps ** 2)
