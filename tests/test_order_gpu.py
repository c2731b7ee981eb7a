"""The spatial order below and above the size where its sort changes, and the tile anchors.

With distinct keys the order is a function of the positions alone, so results
are the same, bit for bit, whatever the input order; chunk edges are multiples
of 256 and the sort changes at 65536.
"""
import numpy as np
import pytest

import nbody_ics
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nb():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    import paper_1803_01190_gb300 as m
    return m


@pytest.mark.parametrize("n", [2, 33, 255, 256, 257, 1025, 8191, 65536, 65537])
def test_order_does_not_depend_on_the_input_order(nb, n):
    pos, _, _ = nbody_ics.uniform_sphere(n, 71 + n)
    mass = nbody_ics.lognormal_masses(n, 72 + n)
    p = np.random.default_rng(n).permutation(n)
    with nb.Simulation(n, "mixed", eps=0.01) as sim:
        a, q = sim.accel(pos, mass)
        b, r = sim.accel(pos[p], mass[p])
    assert np.array_equal(a[p], b) and np.array_equal(q[p], r)


@pytest.mark.parametrize("mode,tol", [("mixed", 2e-6), ("f64e", 1e-12)])
@pytest.mark.parametrize("kind", ["plane", "line", "lattice", "negative"])
def test_tied_coordinates(nb, mode, tol, kind):
    """Coordinates that tie in whole tiles (medians among equal values, equal keys)."""
    n = 3001
    pos, _, mass = nbody_ics.plummer(n, 75)
    if kind == "plane":
        pos[:, 2] = 0.0
    elif kind == "line":
        pos[:, 0] = np.random.default_rng(76).uniform(-1.0, 1.0, n)  # tiles span 0.2
        pos[:, 1:] = 0.25
    elif kind == "lattice":
        pos = np.stack(np.meshgrid(*[np.arange(15.0)] * 3, indexing="ij"), -1).reshape(-1, 3)[:n]
    else:
        pos = -np.abs(pos) - 1.0
    with nb.Simulation(n, mode, eps=0.05) as sim:
        acc, pot = sim.accel(pos, mass)
    oa, op, smag = oracle.accel(pos, mass, 0.05)
    # relative to the sum of the magnitudes of the terms: in one or two
    # dimensions the forces on many particles nearly cancel.  A term d / r^3
    # carries the roundings of x_i - c and x_j - c (u |x - c| each, u = 2^-24,
    # f64e 2^-48), amplified at most 4 times (once in d, three times in r) and
    # divided by r >= eps = |x - c| / 20 where a tile of the core spans 1: 80 u
    err = np.linalg.norm(acc - oa, axis=1) / smag
    assert err.max() <= 80 * (2.0 ** -24 if mode == "mixed" else 2.0 ** -48)
    assert np.sqrt(np.mean(err ** 2)) <= tol
    assert np.abs(pot / op - 1).max() <= 10 * tol


@pytest.mark.parametrize("n", [300, 65536, 65537])
def test_launches_counted(nb, n):
    """One evaluation: pack, the order's own three kernels, prep, force, sums out."""
    pos, _, mass = nbody_ics.plummer(n, 3)
    with nb.Simulation(n, "mixed", eps=0.05) as sim:
        before = sim.launch_count
        sim.accel(pos, mass)
        assert sim.launch_count - before == 7
