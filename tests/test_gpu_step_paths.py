"""Branches of the step on the CUDA path against the oracle: the fixed-point
FP64 collision inside and outside its range, the chained launches of small
lattices (body updates and tile clearing in extra blocks of the fluid kernel)
over group lengths, body counts, substeps and pore axes, fluid kernels that fetch
ahead into L2, rows cut into blocks, fast rotations, and results read from
host-mapped memory after calls that make them stale.

Tolerances as in test_gpu_parity.py: TOL = 1e-12 (FP64) and 1e-5 (FP32) of
w_i rho0 for populations. Populations within TOL give a velocity within TOL / 3
(sum of w_i |c_i| per component); bead forces are gamma u with u ~ 0.01 and more,
so they and what they drive (bodies heavier than 10, at most 29 steps) are held
to 100 TOL, a body's totals relative to its largest bead force times the bead
count, since a few beads can cancel."""
import numpy as np
import pytest

from helpers import Pair, W19, perturbed_populations
from paper_1604_01829_gb300 import workloads as Wl

pytestmark = pytest.mark.gpu

TOL = {64: 1e-12, 32: 1e-5}
MRT = dict(collision=1, gamma_shear=-0.45, gamma_bulk=-0.2, gamma_odd=0.3, gamma_even=-0.1)


@pytest.mark.parametrize("rho0", [1.0, 6.004, 1e-3, 0.4])
@pytest.mark.parametrize("kT", [0.0, 1e-4, 0.02])
@pytest.mark.parametrize("force", [0.0, 1e-5, 0.6])
def test_fp64_collision_in_and_out_of_the_fixed_point_range(rho0, kT, force):
    """Nodes with negative, oversized, tiny and vanishing populations, high speeds
    and low densities beside ordinary ones; kT = 0.02 rho0 and |F| = 0.6 rho0 leave
    the range for every node."""
    params = dict(MRT) if kT else dict(collision=0, tau=0.8)
    P = Pair(18, 7, 6, precision=64, rho0=rho0, kT=kT * rho0, seed=5, body_force=(0.0, 0.3 * force * rho0, force * rho0),
             **params)
    f = perturbed_populations(P.N, rho0=rho0, seed=9)
    rng = np.random.default_rng(2)
    at = rng.permutation(P.N)
    f[rng.integers(1, 19, 40), at[:40]] *= -0.5                    # negative
    f[rng.integers(7, 19, 40), at[40:80]] += 0.2 * rho0             # beyond 1/16
    f[0, at[80:100]] += 0.4 * rho0                                  # beyond 1/2
    f[rng.integers(1, 19, 40), at[100:140]] = 1e-12 * rho0          # far below the grid's steps
    f[rng.integers(1, 19, 40), at[140:180]] = 0.0
    f[1, at[180:200]] += 0.11 * rho0                                # fast
    f[:, at[200:210]] *= 0.2                                        # thin
    P.set_populations(f)
    P.step(1)
    assert P.pop_error() <= 1e-12 * (1 + force)


@pytest.mark.parametrize("size", [(150, 97, 97), (33, 211, 205), (4100, 19, 18), (2, 840, 841)])
@pytest.mark.parametrize("case", ["noise", "mrt", "bgk"])
def test_fetching_ahead(size, case):
    """FP32 boxes just above the size from which the fluid kernel fetches ahead,
    with rows that are no multiple of its lines or blocks."""
    params = dict(MRT, kT=1e-4, seed=2) if case == "noise" else (dict(MRT) if case == "mrt" else dict(collision=0, tau=0.8))
    P = Pair(*size, precision=32, body_force=(1e-5, 0, 2e-5), **params)
    P.set_populations(perturbed_populations(P.N, amp=0.005, u_amp=0.01, seed=8))
    P.step(3)
    assert P.pop_error() <= TOL[32]


@pytest.mark.parametrize("tile,order", [(128, 0), (64, 0), (256, 1), (128, 2)])
def test_batch_fetching_ahead(tile, order):
    """A batch above that size: instances of odd sizes, a pore among them, against
    the oracle."""
    from oracle import oracle as O
    from paper_1604_01829_gb300 import lb
    sizes = [(61, 43, 67), (67, 71, 59), (64, 64, 64), (71, 67, 73), (33, 95, 101)]
    pars = [dict(nx=n[0], ny=n[1], nz=n[2], precision=32, body_force=(0, 1e-5, 1e-5), **MRT) for n in sizes]
    B = lb.LBBatch(pars)
    B.lb_batch_set_pore(3, 30.0, 2)
    B.lb_batch_set_schedule(tile, 4, order)
    orcs = []
    for k, n in enumerate(sizes):
        f = perturbed_populations(n[0] * n[1] * n[2], amp=0.005, u_amp=0.01, seed=k)
        B.lb_batch_set_populations(k, f)
        o = O.OracleLB(*n, body_force=(0, 1e-5, 1e-5), **MRT)
        if k == 3:
            o.set_pore(30.0, 2)
        o.set_populations(f)
        orcs.append(o)
    B.lb_batch_step(3)
    for k, o in enumerate(orcs):
        o.step(3)
        fluid = o.mask == 0 if k == 3 else slice(None)
        d = B.lb_batch_get_populations(k)[:, fluid] - o.populations()[:, fluid]
        assert np.max(np.abs(d) / W19[:, None]) <= TOL[32]


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("nx", [129, 150, 190, 224])
def test_rows_split_without_waste(nx, precision):
    """Rows longer than a block, cut into 128, 64 or 32 threads."""
    P = Pair(nx, 7, 5, precision=precision, gamma_bead=0.05, **MRT)
    P.set_populations(perturbed_populations(P.N, amp=0.005, u_amp=0.01, seed=nx))
    P.add_body(Wl.fibonacci_sphere(12, 1.5), [nx - 0.7, 6.8, 0.2], mass=30.0, inertia=(40, 40, 40), F_ext=(1e-3, 0, 0))
    P.step(5)
    assert P.pop_error() <= TOL[precision]


def _beads(rng, n):
    return rng.uniform(-2.0, 2.0, (n, 3))


def _force_errors(P, b):
    g, o = P.gpu.lb_forces(b, per_bead=True), P.orc.body(b)
    pb = P.orc.bead_forces(b)
    scale = np.abs(pb).max() * len(pb)
    return max(np.abs(g[0] - o["F"]).max() / scale, np.abs(g[1] - o["T"]).max() / (3 * scale),
               np.abs(g[2] - pb).max() / np.abs(pb).max())


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("nbodies,nbeads,substeps", [(1, 1, 1), (1, 300, 2), (5, 7, 1), (70, 3, 3), (130, 2, 1)])
def test_chained_steps(precision, nbodies, nbeads, substeps):
    rng = np.random.default_rng(nbodies)
    P = Pair(21, 18, 19, precision=precision, kT=1e-4, seed=3, gamma_bead=0.05, md_substeps=substeps, compensate_force=1, **MRT)
    P.set_populations(perturbed_populations(P.N, amp=0.005, u_amp=0.01, seed=4))
    for b in range(nbodies):
        P.add_body(_beads(rng, nbeads), rng.random(3) * (21, 18, 19), rng.standard_normal(4), mass=20.0, inertia=(30, 35, 42),
                   F_ext=1e-3 * rng.standard_normal(3), T_ext=1e-3 * rng.standard_normal(3), fixed=b % 3 if nbodies > 1 else 0)
    for n in (1, 2, 8, 5, 13):                                     # single, short, octet, odd start, mixed
        P.step(n)
    assert P.pop_error() <= TOL[precision]
    for b in range(nbodies):
        e = P.body_errors(b)
        assert max(e["X"], e["V"], e["q"], e["w"], _force_errors(P, b)) <= 100 * TOL[precision]


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_chained_pore_steps(precision, axis):
    n = [19, 20, 21]
    P = Pair(*n, precision=precision, pore=(8.0, axis), gamma_bead=0.05, body_force=(1e-5, 1e-5, 1e-5), **MRT)
    P.set_populations(perturbed_populations(P.N, amp=0.005, u_amp=0.01, seed=6))
    P.add_body(Wl.sphere_raspberry(2.0), np.array(n) / 2 + 0.3, mass=33.0, inertia=(50, 50, 50), F_ext=(1e-3, 0, 2e-3))
    P.step(11)
    assert P.pop_error() <= TOL[precision]
    e = P.body_errors(0)
    assert max(e["X"], e["V"], e["q"], e["w"]) <= 100 * TOL[precision]


@pytest.mark.parametrize("speed", [1e-9, 0.3, 0.99, 1.01, 3.0])
def test_fast_rotation(speed):
    """Half angles on both sides of 1/2, where the power series ends."""
    P = Pair(16, 16, 16, precision=64, gamma_bead=0.01, collision=0, tau=0.9)
    w = speed * np.array([0.6, -0.48, 0.64])
    P.add_body(Wl.fibonacci_sphere(12, 2.0), [8.2, 7.9, 8.1], mass=40.0, inertia=(60, 80, 110), w=w, F_ext=(1e-4, 0, 0))
    P.step(6)
    e = P.body_errors(0)
    assert max(e["X"], e["V"], e["q"], e["w"]) <= 1e-11
    assert P.pop_error() <= 1e-11                                  # speeds of 3 w per unit of population


def test_mapped_results_follow_the_state():
    from paper_1604_01829_gb300 import lb
    kw = dict(precision=64, gamma_bead=0.05, collision=0, tau=0.9)
    h = lb.LB(16, 16, 16, **kw)
    h.lb_add_raspberry(Wl.sphere_raspberry(2.0), [8.2, 7.9, 8.1], mass=33.0, inertia=(50, 50, 50), F_ext=(1e-3, 0, 0))
    h.lb_step(5)
    F, T = h.lb_forces_all()
    assert np.array_equal(F, h.lb_forces(0)[0]) and np.array_equal(T, h.lb_forces(0)[1])
    data, at5 = h.lb_checkpoint_save(), h.lb_get_body(0)
    h.lb_set_body_state(0, X=(3.0, 4.0, 5.0))
    assert np.array_equal(h.lb_get_body(0)["X"], [3.0, 4.0, 5.0]) and np.array_equal(h.lb_get_body(0)["V"], at5["V"])
    h.lb_step(4)
    assert np.abs(h.lb_get_body(0)["X"] - [3.0, 4.0, 5.0]).max() < 0.1
    h.lb_checkpoint_load(data)
    assert all(np.array_equal(h.lb_get_body(0)[k], at5[k]) for k in at5)
    assert np.array_equal(h.lb_forces_all()[0], F)

    B = lb.LBBatch([dict(nx=16, ny=16, nz=16 + k, **kw) for k in range(3)])
    for k in range(3):
        B.lb_batch_add_raspberry(k, Wl.sphere_raspberry(2.0), [8.2, 7.9, 8.1], mass=33.0, inertia=(50, 50, 50),
                                 F_ext=(1e-3, 0, 1e-4 * k))
    before = B.lb_batch_get_body(2)["X"]
    assert np.array_equal(before, [8.2, 7.9, 8.1])
    for n in (1, 8, 3, 10):
        B.lb_batch_step(n)
    data = B.lb_batch_checkpoint_save()
    got = [(B.lb_batch_get_body(k), B.lb_batch_forces(k)) for k in range(3)]
    B.lb_batch_autotune(2)
    for k in range(3):
        body, (F, T) = B.lb_batch_get_body(k), B.lb_batch_forces(k)
        assert all(np.array_equal(body[q], got[k][0][q]) for q in body)
        assert np.array_equal(F, got[k][1][0]) and np.array_equal(T, got[k][1][1])
    B.lb_batch_step(6)
    assert not np.array_equal(B.lb_batch_get_body(1)["X"], got[1][0]["X"])
    B.lb_batch_checkpoint_load(data)
    assert np.array_equal(B.lb_batch_get_body(1)["X"], got[1][0]["X"])
    assert np.array_equal(B.lb_batch_forces(1)[0], got[1][1][0])


@pytest.mark.parametrize("gap", [2.0 ** -50, 1e-12, 2.0 ** -33, 2.0 ** -31, 2.0 ** -30, 1e-8])
@pytest.mark.parametrize("case", ["bgk", "mrt", "noise"])
def test_fp64_rates_close_to_minus_one(gap, case):
    """Rates down to the closest to -1 that are accepted (tau - 1/2 = gap / 4),
    where the weight of the equilibrium moments is 1/2 and its fixed-point form
    ends; single lattices and batches."""
    from paper_1604_01829_gb300 import lb
    g = -1.0 + gap
    params = (dict(collision=0, tau=0.5 + 0.25 * gap) if case == "bgk"
              else dict(MRT, gamma_shear=g, kT=1e-4 if case == "noise" else 0.0, seed=3))
    P = Pair(13, 7, 6, precision=64, body_force=(0.0, 1e-5, 0.0), **params)
    f = perturbed_populations(P.N, seed=11)
    P.set_populations(f)
    P.step(1)
    assert P.pop_error() <= TOL[64]
    B = lb.LBBatch([dict(nx=13, ny=7, nz=6, precision=64, body_force=(0.0, 1e-5, 0.0), **params)])
    B.lb_batch_set_populations(0, f)
    B.lb_batch_step(1)
    o = P.orc.populations()
    assert np.max(np.abs(B.lb_batch_get_populations(0) - o) / W19[:, None]) <= TOL[64]


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("axis,spacing,rp,rr", [(0, 40.0, 3.0, 3.0), (1, 7.0, 6.0, 2.0), (2, 1.5, 2.5, 2.5), (1, 0.7, 1.0, 1.0),
                                                (0, 3.0, 0.5, 0.9)])
def test_wall_beads_shared_by_a_beads_lanes(axis, spacing, rp, rr, precision):
    """Windows of three wall beads, of a few columns, of hundreds, and the whole
    ring and row; most of the raspberry's beads within reach of the wall."""
    n = [19, 19, 19]
    n[axis] = 14
    P = Pair(*n, precision=precision, pore=(8.0, axis), gamma_bead=0.02, **MRT)
    P.gpu.lb_set_pore_beads(spacing, rp, rr, 1e-4)
    P.orc.set_pore_beads(8.0, axis, spacing, rp, rr, 1e-4)
    P.set_populations(perturbed_populations(P.N, amp=0.005, u_amp=0.01, seed=axis))
    X = np.array(n) / 2 + 0.2
    X[(axis + 1) % 3] += 2.4
    beads = Wl.sphere_raspberry(5.0)
    P.add_body(beads, X, mass=5e4, inertia=(5e5, 5.2e5, 5.4e5))
    near = sum(np.linalg.norm(P.orc.wall_force(x)) > 0 for x in X + beads)
    assert near >= 5
    P.step(3)
    assert P.pop_error() <= TOL[precision]
    e = P.body_errors(0)
    assert max(e["X"], e["V"], e["q"], e["w"], _force_errors(P, 0)) <= 100 * TOL[precision]


@pytest.mark.parametrize("kT", [1.9e-3, 2.0e-3, 2.1e-3, 9e-3])
def test_fp64_noise_on_both_sides_of_the_fixed_point_rule(kT):
    """kT = 0.002 rho0, where a lattice changes to the FP64 evaluation; below it
    nodes that the noise takes out of range, beside ordinary ones."""
    P = Pair(17, 9, 8, precision=64, rho0=1.3, kT=kT * 1.3, seed=4, body_force=(0.0, 1e-5, 0.0), **MRT)
    P.set_populations(perturbed_populations(P.N, rho0=1.3, seed=12))
    P.step(4)
    assert P.pop_error() <= TOL[64]
