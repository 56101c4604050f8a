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
