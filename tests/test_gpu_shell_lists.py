"""The automatic pair search of the shell construction (per-bead neighbour
lists, Newton surface roots) against the oracle and the all-pairs search.

Tolerances as for the other searches (test_gpu_shell.py): the lists sum the
same pairs in the same order and only the rounding of the surface root
differs."""
import numpy as np
import pytest

from oracle import construction as C

pytestmark = pytest.mark.gpu

TOL = {64: 1e-9, 32: 1e-5}


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("n", [1, 2, 33, 512, 513, 1024, 1025, 1700, 2049, 2600])
def test_lists_equal_all_pairs(n, precision):
    """Edges of the beads-per-thread layouts and, at 2600, the size beyond
    which lists do not fit."""
    from paper_1604_01829_gb300 import lb, workloads as W
    a = max(1.0, np.sqrt(n / (4 * np.pi)))
    ax = (1.2 * a, a, 0.9 * a)
    X0 = W.random_shell_start(*ax, n, seed=n, spread=0.0) if n < 3 else W.spread_shell_start(*ax, n, seed=n, jitter=0.02)
    got = [lb.lb_relax_shells([ax], [X0], steps=40, precision=precision, project_final=False, pair_search=s)[0]
           for s in (0, 1)]
    assert np.abs(got[0] - got[1]).max() <= TOL[precision]


@pytest.mark.parametrize("precision", [64, 32])
def test_lists_match_oracle_while_beads_move_far(precision):
    """Beads started 30 % off the surface and crowded: many list rebuilds."""
    from paper_1604_01829_gb300 import lb, workloads as W
    for ax in ((3.0, 3.0, 3.0), (6.0, 2.5, 2.5), (2.0, 4.0, 3.0)):
        X0 = W.spread_shell_start(*ax, int(0.5 * W.ellipsoid_area(*ax)), seed=9, jitter=0.3)
        (X,) = lb.lb_relax_shells([ax], [X0], steps=150, dt=0.01, eta=100.0, precision=precision, project_final=False)
        ref = C.relax_shell(X0, ax, 150, dt=0.01, eta=100.0, project_final=False)
        assert np.abs(X - ref).max() <= TOL[precision]
        assert np.abs(X - X0).max() > 0.3


def test_a_list_that_overflows_tests_all_pairs():
    """Six beads per unit area: about 70 within the list radius, more than a list holds."""
    from paper_1604_01829_gb300 import lb, workloads as W
    ax = (3.0, 3.0, 3.0)
    X0 = W.spread_shell_start(*ax, int(6 * W.ellipsoid_area(*ax)), seed=4)
    got = [lb.lb_relax_shells([ax], [X0], steps=20, dt=1e-5, eta=1e5, precision=64, project_final=False,
                              pair_search=s)[0] for s in (0, 1)]
    assert np.abs(got[0] - got[1]).max() <= 1e-9


def test_beads_without_a_unique_nearest_point():
    """At the centre, on the medial plane and on an axis inside: as the bisection places them."""
    from paper_1604_01829_gb300 import lb
    ax = (4.0, 3.0, 2.0)
    X0 = np.array([[0, 0, 0], [1.0, 0.5, 0], [0, 0, 1.0], [3.9, 0, 0], [0.1, 0, 0], [0, 2.0, 1e-9], [9.0, 8.0, 7.0]])
    got = [lb.lb_relax_shells([ax], [X0 + 0.0], steps=3, dt=1e-3, eta=1000.0, sigma=0.01, epsilon=1e-6, precision=64,
                              project_final=False, pair_search=s)[0] for s in (0, 1)]
    assert np.abs(got[0] - got[1]).max() <= 1e-9


def test_many_shells_equal_each_alone():
    from paper_1604_01829_gb300 import lb, workloads as W
    rng = np.random.default_rng(6)
    axes = [tuple(rng.uniform(1.5, 6.0, 3)) for _ in range(30)]
    starts = [W.spread_shell_start(*ax, int(rng.integers(5, 300)), seed=60 + s) for s, ax in enumerate(axes)]
    together = lb.lb_relax_shells(axes, starts, steps=60, precision=32)
    for s in (0, 11, 29):
        assert np.array_equal(lb.lb_relax_shells([axes[s]], [starts[s]], steps=60, precision=32)[0], together[s])


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("n,density", [(32, 6.0), (33, 6.0), (200, 6.0), (255, 2.3), (255, 2.6), (900, 6.0), (1100, 3.0), (2000, 6.0),
                                       (4, 100.0), (600, 100.0)])
def test_crowded_shells(n, density, precision):
    """Both sides of the density from which lists are longer (24 beads in the list
    radius: 2.4 a unit area), up to lists of every other bead: as all pairs."""
    from paper_1604_01829_gb300 import lb, workloads as W
    a = np.sqrt(n / density / (4 * np.pi))
    X0 = W.spread_shell_start(a, a, a, n, seed=n)
    # small steps: 20 of them stay far from the chaos of a shell that blows up
    dt = 1e-6 if density < 50 else 1e-12
    got = [lb.lb_relax_shells([(a, a, a)], [X0], steps=20, dt=dt, eta=1.0 / dt, precision=precision, project_final=False,
                              pair_search=s)[0] for s in (0, 1)]
    assert np.abs(got[0] - got[1]).max() <= TOL[precision]


@pytest.mark.parametrize("precision", [64, 32])
def test_crowded_and_loose_shells_together(precision):
    """Shells with short and long lists in one call as each alone: bit for bit in
    FP32, in FP64 to the rounding of kernels that carry 1 or 2 beads a thread."""
    from paper_1604_01829_gb300 import lb, workloads as W
    axes, starts = [], []
    for n, density in ((300, 1.0), (300, 6.0), (40, 3.0), (700, 2.0), (700, 3.5)):
        a = np.sqrt(n / density / (4 * np.pi))
        axes.append((a, a, a))
        starts.append(W.spread_shell_start(a, a, a, n, seed=n))
    kw = dict(steps=30, dt=1e-6, eta=1e6, precision=precision)
    together = lb.lb_relax_shells(axes, starts, **kw)
    for s in range(5):
        alone = lb.lb_relax_shells([axes[s]], [starts[s]], **kw)[0]
        assert np.abs(alone - together[s]).max() <= (1e-12 if precision == 64 else 0.0)


@pytest.mark.parametrize("precision", [64, 32])
def test_a_clump_on_a_loose_shell(precision):
    """45 beads within one list radius of each other on a shell of one bead a unit
    area: more than a list holds, the others' lists do."""
    from paper_1604_01829_gb300 import lb, workloads as W
    a = 6.0
    X0 = W.spread_shell_start(a, a, a, 400, seed=3)
    rng = np.random.default_rng(5)
    X0[100:145] = X0[7] + 0.4 * rng.standard_normal((45, 3))
    got = [lb.lb_relax_shells([(a, a, a)], [X0], steps=20, dt=1e-8, eta=1e8, precision=precision, project_final=False,
                              pair_search=s)[0] for s in (0, 1)]
    assert np.abs(got[0] - got[1]).max() <= TOL[precision]
