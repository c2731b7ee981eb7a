"""F64E: both sides of a pair are taken from the tile's anchor in binary64.

A system far from the origin keeps the accuracy of one at it: coordinates are
off by 2^-49 of their distance from the anchor, not of their magnitude.
"""
import numpy as np
import pytest

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


@pytest.mark.parametrize("n", [2, 257, 700, 2049])
@pytest.mark.parametrize("sym", [0, 1])
@pytest.mark.parametrize("equal", [True, False])
def test_far_from_the_origin(nb, n, sym, equal):
    rng = np.random.default_rng(n)
    pos = np.array([4096.0, -3000.0, 1.0e4]) + rng.random((n, 3))
    mass = np.full(n, 1.0 / n) if equal else rng.uniform(0.5, 2.0, n) / n
    eps = 0.05
    with nb.Simulation(n, "f64e", eps=eps) as sim:
        sim.set_symmetric(sym if n > 256 else 0)
        acc, pot = sim.accel(pos, mass)
    oa, op, _ = oracle.accel(pos, mass, eps)
    # |x - c| < 1: each coordinate of a difference is off by at most 2^-49 from
    # either split and 2^-47 from adding the low parts, 2.5e-14 in all three; a
    # term m d / r^3 changes by at most 4 m / r^3 of that, m / r by m / r^2, and
    # the float-float arithmetic adds 2^-43 of a term
    r2 = ((pos[:, None] - pos[None]) ** 2).sum(2) + eps * eps
    np.fill_diagonal(r2, np.inf)
    bound = (mass / r2 ** 1.5).sum(1) * 1e-13 + (mass / r2).sum(1) * 2.0 ** -43
    assert (np.linalg.norm(acc - oa, axis=1) <= bound).all()
    bound = (mass / r2).sum(1) * 2.5e-14 + (mass / r2 ** 0.5).sum(1) * 2.0 ** -43
    assert (np.abs(pot - op) <= bound).all()


@pytest.mark.parametrize("equal", [True, False])
def test_potential_sums_each_pair_once(nb, equal):
    """Coordinates that float-floats hold exactly leave the error of the sums.  With the
    sums renormalised at every term its RMS over these draws is 1.66e-15 (1.64e-15 for
    uneven masses), at every second step 1.82e-15 (1.81e-15)."""
    err = []
    for s in range(5):
        rng = np.random.default_rng(s)
        pos = rng.integers(-64, 65, (1500, 3)) * 1.0
        mass = np.ones(1500) if equal else rng.integers(1, 2 ** 20, 1500) * 2.0 ** -20
        with nb.Simulation(1500, "f64e", eps=64.0) as sim:
            sim.set_symmetric(1)
            _, pot = sim.accel(pos, mass)
        _, op, _ = oracle.accel(pos, mass, 64.0)
        err.append(np.sqrt((((pot - op) / op) ** 2).mean()))
    assert np.mean(err) <= 1.74e-15
