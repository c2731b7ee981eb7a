"""The fixed-point pair sums of the binary64 mode (softened systems), at the edges of their rules.

The reference is the FP64 oracle.  A tile that the fixed-point form does not
take, and pairs too close for its unit, run in binary64, so every case has to
meet the same gate: |da| <= 1e-12 |a| + 4 u sqrt(N) S (tests/gates.py), and
potentials to 1e-12.
"""
import numpy as np
import pytest

import nbody_ics
import oracle
from gates import fp64_accel_gate

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


def _case(kind, n):
    pos, _, mass = nbody_ics.plummer(n, 20180300 + n)
    eps = 0.01
    if kind == "offset":  # coordinates far larger than the differences
        pos = pos + np.array([3.0e6, -7.0e5, 1.0])
    elif kind == "scaled":  # units of 1e-40 and 1e30
        pos, eps, mass = pos * 1e-40, eps * 1e-40, mass * 1e30
    elif kind == "close":  # half the particles within 1e-5 of another, one escaper
        pos[n // 2:n // 2 * 2] = pos[:n // 2] + 1e-5 * np.random.default_rng(1).standard_normal((n // 2, 3))
        pos[-1] = [4.0e3, 0.0, 0.0]
        eps = 1e-6
    elif kind == "masses":  # over the mass rule in some tiles, zeros, within it in others
        rng = np.random.default_rng(2)
        mass = mass * np.exp(0.5 * rng.standard_normal(n))
        mass[: n // 3] *= np.exp2(rng.uniform(-30, 30, n // 3))
        mass[n // 2:n // 2 + 40] = 0.0
    elif kind == "coincident":
        pos[1::2] = pos[::2][: len(pos[1::2])]
    elif kind == "wide eps":
        eps = 300.0
    return pos, mass, eps


KINDS = ["plain", "offset", "scaled", "close", "masses", "coincident", "wide eps"]


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("n", [2, 127, 129, 1000, 2305])
@pytest.mark.parametrize("ipt", [1, 2, 8])
def test_one_sided(nb, kind, n, ipt):
    pos, mass, eps = _case(kind, n)
    with nb.Simulation(n, "fp64", eps=eps) as sim:
        sim.set_symmetric(0)
        sim.set_launch(ipt, 0)
        acc, pot = sim.accel(pos, mass)
    _check(pos, mass, eps, acc, pot)


# blocks of 256: n = 257, 512 (M = 2), 700 (M = 3), 2305 (M = 10, tail of one)
@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("n", [257, 512, 700, 2305])
def test_each_pair_once(nb, kind, n):
    pos, mass, eps = _case(kind, n)
    with nb.Simulation(n, "fp64", eps=eps) as sim:
        sim.set_symmetric(1)
        acc, pot = sim.accel(pos, mass)
    _check(pos, mass, eps, acc, pot)


def _check(pos, mass, eps, acc, pot):
    oa, op, smag = oracle.accel(pos, mass, eps)
    ok, err, amag = fp64_accel_gate(acc, oa, smag, len(mass))
    assert ok.all(), float((err / np.maximum(amag, 1e-300)).max())
    assert np.all(np.abs(pot - op) <= 1e-12 * np.abs(op))


@pytest.mark.parametrize("mode", ["fp64", "f64e", "mixed", "fp32"])
@pytest.mark.parametrize("n", [1500, 20003])
def test_rows_of_equal_masses(nb, mode, n):
    """Row blocks that start inside i-blocks, with tiles of equal masses: bit for bit
    the rows of one evaluation, whichever rows share a block."""
    pos, _, mass = nbody_ics.plummer(n, 20180400)
    with nb.Simulation(n, mode, eps=0.02) as sim:
        if mode in ("fp64", "f64e"):
            sim.set_symmetric(0)
        if mode != "fp32":
            sim.set_order("input")
        acc, pot = sim.accel(pos, mass)
        for i0, ni in ((0, 1), (1, n - 1), (333, 700), (n - 77, 77)):
            a, p = sim.accel_rows(i0, ni, pos, mass)
            assert np.array_equal(a, acc[i0:i0 + ni]) and np.array_equal(p, pot[i0:i0 + ni])


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("where", ["pos", "mass"])
def test_non_finite_input_gives_non_finite_output(nb, bad, where):
    pos, mass, eps = _case("plain", 300)
    (pos if where == "pos" else mass[:, None])[17, 0] = bad
    with nb.Simulation(300, "fp64", eps=eps) as sim:
        acc, pot = sim.accel(pos, mass)
    others = np.delete(np.arange(300), 17)
    if np.isnan(bad) or where == "mass":
        assert not np.isfinite(acc[others]).any() and not np.isfinite(pot[others]).any()
    else:  # at an infinite distance: no force, by inf * 0
        assert not np.isfinite(acc[others, 0]).any()


def test_subnormal_masses(nb):
    # below the fixed-point form's masses: binary64, whose subnormal results are exact to
    # a few units of 2^-1074
    pos, mass, _ = _case("plain", 300)
    mass = np.full(300, 3.0e-310)
    for sym in (0, 1):
        with nb.Simulation(300, "fp64", eps=0.5) as sim:
            sim.set_symmetric(sym)
            acc, pot = sim.accel(pos, mass)
        oa, op, _ = oracle.accel(pos, mass, 0.5)
        assert np.abs(acc).max() > 1e-309
        assert np.abs(acc - oa).max() <= 300 * 2.0 ** -1073
        assert np.abs(pot - op).max() <= 300 * 2.0 ** -1073


def test_negative_mass(nb):
    pos, mass, eps = _case("plain", 300)
    mass[5] = -mass[5]
    with nb.Simulation(300, "fp64", eps=eps) as sim:
        acc, pot = sim.accel(pos, mass)
    a1, p1, _ = oracle.accel(pos, np.maximum(mass, 0.0), eps)
    a2, p2, _ = oracle.accel(pos, np.maximum(-mass, 0.0), eps)
    assert np.abs(acc - (a1 - a2)).max() <= 1e-12 * np.abs(a1).max()
    assert np.abs(pot - (p1 - p2)).max() <= 1e-12 * np.abs(p1).max()


# A tile that the fixed point does not take must leave the ones after it alone: the
# first half of a column block holds a tracer far below the other masses, the second
# half none
@pytest.mark.parametrize("masses", ["light", "heavy", "one mass"])
@pytest.mark.parametrize("tracer", [1e-25, 0.5, -1.0])
@pytest.mark.parametrize("n", [512, 1000])
def test_tile_after_a_refused_one(nb, masses, tracer, n):
    pos, mass, eps = _case("plain", n)
    rng = np.random.default_rng(n)
    if masses == "light":
        mass = 1e-5 * rng.uniform(1.0, 9.0, n)
    elif masses == "heavy":
        mass = np.exp2(rng.uniform(0.0, 6.0, n)) * 100
    mass[256 + 10] = tracer * mass[0]
    with nb.Simulation(n, "fp64", eps=eps) as sim:
        sim.set_symmetric(1)
        acc, pot = sim.accel(pos, mass)
    if tracer > 0:
        _check(pos, mass, eps, acc, pot)
    else:  # the oracle takes no negative masses: the sum of both signs' parts
        (a1, p1, s1), (a2, p2, s2) = (oracle.accel(pos, np.maximum(q, 0.0), eps) for q in (mass, -mass))
        ok, err, _ = fp64_accel_gate(acc, a1 - a2, s1 + s2, n)
        assert ok.all() and np.all(np.abs(pot - (p1 - p2)) <= 1e-12 * (np.abs(p1) + np.abs(p2)))


# r^2 + eps^2 exactly a power of four, where 1/r is at the top of its range: lattices
# whose (1,1,1) or (1,0,0) neighbours have it, particles at one place
@pytest.mark.parametrize("kind,eps", [("lattice", 1.0), ("lattice", 1e-12), ("coincident", 0.25)])
@pytest.mark.parametrize("sym", [0, 1])
def test_distances_that_are_powers_of_two(nb, kind, eps, sym):
    if kind == "lattice":
        pos = np.stack(np.meshgrid(*[np.arange(12.0)] * 3), -1).reshape(-1, 3)
    else:
        pos = np.tile(np.random.default_rng(3).integers(-4, 5, (256, 3)) * 1.0, (4, 1))
    mass = np.full(len(pos), 0.5)
    with nb.Simulation(len(pos), "fp64", eps=eps) as sim:
        sim.set_symmetric(sym)
        acc, pot = sim.accel(pos, mass)
    _check(pos, mass, eps, acc, pot)


@pytest.mark.parametrize("bits", [9, 12, 20, 30, 40])
@pytest.mark.parametrize("where", ["alone", "at a light one"])
@pytest.mark.parametrize("sym", [0, 1])
def test_heavy_particle(nb, bits, where, sym):
    """The forces of the light particles alone: on the heavy one itself, and on a
    light one at the heavy one's place, where its force vanishes."""
    n = 1000
    pos, mass, eps = _case("plain", n)
    mass[:] = 2.0 ** -bits
    mass[5] = 1.0
    if where != "alone":
        pos[700] = pos[5]
    with nb.Simulation(n, "fp64", eps=eps) as sim:
        sim.set_symmetric(sym)
        acc, pot = sim.accel(pos, mass)
    _check(pos, mass, eps, acc, pot)
    # no less exact than binary64 terms: 2^-53 of each, twice over, whatever their order
    oa, _, smag = oracle.accel(pos, mass, eps)
    assert np.linalg.norm(acc[5] - oa[5]) <= 2.0 ** -52 * smag[5]


# Separations far below the softening: of the whole system, or inside two clumps that
# are far apart in units of it
@pytest.mark.parametrize("size", [2.0 ** -7, 1e-3, 1e-4, 1e-6])
@pytest.mark.parametrize("apart", [0.0, 32.0, 512.0, 1000.0])
@pytest.mark.parametrize("sym", [0, 1])
def test_separations_below_the_softening(nb, size, apart, sym):
    n = 700
    pos = size * np.random.default_rng(4).standard_normal((n, 3))
    pos[1::2, 0] += apart
    mass = np.full(n, 1.0 / n)
    with nb.Simulation(n, "fp64", eps=1.0) as sim:
        sim.set_symmetric(sym)
        acc, pot = sim.accel(pos, mass)
    _check(pos, mass, 1.0, acc, pot)


# Far particles in every tile, so that most, some or few of the other pairs are too close for
# the tiles' units (within 2^-10 of the extent)
@pytest.mark.parametrize("extent", [30.0, 300.0, 1e3, 1e4, 1e8])
@pytest.mark.parametrize("equal", [True, False])
@pytest.mark.parametrize("n,sym", [(129, 0), (1000, 0), (9001, 0), (257, 1), (1000, 1), (2305, 1)])
def test_far_particles(nb, extent, equal, n, sym):
    pos, mass, eps = _case("plain", n)
    rng = np.random.default_rng(n)
    v = rng.standard_normal((len(pos[7::50]), 3))
    pos[7::50] = extent * v / np.linalg.norm(v, axis=1)[:, None]
    if not equal:
        mass = mass * rng.uniform(0.5, 1.0, n)
        mass[n // 3] *= 2.0 ** -30  # one tile outside the mass rule as well
    with nb.Simulation(n, "fp64", eps=eps) as sim:
        sim.set_symmetric(sym)
        acc, pot = sim.accel(pos, mass)
    _check(pos, mass, eps, acc, pot)


# A softening above the system's size and a spread of masses take digits from the same
# terms.  No more is lost than binary64 terms may lose: 2 of 3 roundings (2^-53 each) of a
# term and as much again for the additions of a hundred of them
@pytest.mark.parametrize("bits", [1, 3, 5, 8])
@pytest.mark.parametrize("size", [2.0 ** -2, 2.0 ** -5, 2.0 ** -7, 2.0 ** -9])
@pytest.mark.parametrize("offset", [0.0, 2.0 ** 20])
@pytest.mark.parametrize("n,sym", [(100, 0), (300, 1)])
def test_masses_below_a_large_softening(nb, bits, size, offset, n, sym):
    rng = np.random.default_rng(bits)
    pos = offset * size + size * rng.standard_normal((n, 3))
    mass = np.full(n, 2.0 ** -bits)
    mass[n // 2] = 1.0
    with nb.Simulation(n, "fp64", eps=1.0) as sim:
        sim.set_symmetric(sym)
        acc, pot = sim.accel(pos, mass)
    _check(pos, mass, 1.0, acc, pot)
    oa, _, smag = oracle.accel(pos, mass, 1.0)
    assert (np.linalg.norm(acc - oa, axis=1) <= 2.0 ** -50 * smag).all()
