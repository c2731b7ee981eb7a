"""Tiles of equal masses in the binary32 modes and F64E: leaving the mass out of the pair body.

The rules (masses up to 1, in FP32 powers of two; a softening that keeps 1/r^3
finite) send everything else through the body with the mass.
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

TOL = {"f64e": 1e-11, "mixed": 1e-5, "fp32": 1e-4}


@pytest.fixture(scope="module")
def nb():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    import paper_1803_01190_gb300 as m
    return m


def _errors(nb, mode, pos, mass, eps, sym=0):
    with nb.Simulation(len(mass), mode, eps=eps) as sim:
        if mode == "f64e":
            sim.set_symmetric(sym)
        acc, pot = sim.accel(pos, mass)
    oa, op, _ = oracle.accel(pos, mass, eps)
    return (np.linalg.norm(acc - oa) / np.linalg.norm(oa), np.linalg.norm(pot - op) / np.linalg.norm(op))


# lengths and masses: around 1; in m and kg; where 1/r^3 alone would overflow binary32
UNITS = [(1.0, 1.0 / 1024), (1.0, 1.0), (1.0, 2.0), (1.0, 1.0 / 1000), (1e10, 2.0 ** 100),
         (1e-12, 1e-6)]


@pytest.mark.parametrize("mode", ["f64e", "mixed", "fp32"])
@pytest.mark.parametrize("length,m", UNITS)
@pytest.mark.parametrize("sym", [0, 1])
def test_units(nb, mode, length, m, sym):
    rng = np.random.default_rng(5)
    pos, eps = length * rng.standard_normal((1200, 3)), 0.05 * length
    mass = np.full(1200, m)
    if sym and mode != "f64e":
        pytest.skip("each pair once is a binary64-class path")
    ea, ep = _errors(nb, mode, pos, mass, eps, sym)
    assert ea <= TOL[mode] and ep <= TOL[mode]


@pytest.mark.parametrize("n", [256, 511, 2048, 5000])
def test_fp32_units_do_not_change_the_sums(nb, n):
    """Tiles in and out of units of their mass, in one sum: with masses scaled by a
    power of two out of the rule's range, every tile keeps its mass in the body
    and the sums are the same bits, scaled."""
    rng = np.random.default_rng(n)
    pos = rng.standard_normal((n, 3))
    mass = 2.0 ** rng.integers(-12, -8, (n + 255) // 256)[np.arange(n) // 256]
    mass[n // 3:n // 3 + 5] = 3.0 / 4096
    with nb.Simulation(n, "fp32", eps=0.01) as sim:
        a, p = sim.accel(pos, mass)
        b, q = sim.accel(pos, mass * 2.0 ** 13)
    assert (a * 2.0 ** 13 == b).all() and (p * 2.0 ** 13 == q).all()


@pytest.mark.parametrize("heavy", [1.0, 1e20, 1e32])
@pytest.mark.parametrize("n", [1024, 20000])
def test_fp32_heavy_particle_before_light_tiles(nb, heavy, n):
    """Sums that a heavy particle has made large stay finite in units of a small mass."""
    rng = np.random.default_rng(n)
    pos = rng.standard_normal((n, 3))
    mass = np.full(n, 2.0 ** -40)
    mass[3] = heavy
    ea, ep = _errors(nb, "fp32", pos, mass, 0.05)
    assert ea <= TOL["fp32"] and ep <= TOL["fp32"]


@pytest.mark.parametrize("n", [300, 1200])
@pytest.mark.parametrize("equal", [True, False])
def test_mixed_subnormal_forces(nb, n, equal):
    """Sums below binary32's normal numbers keep what its subnormal ones hold: m y, m y^3
    and d m y^3 of a term and its additions are each off by up to 2^-150, with y <= 2 and
    d y^2 <= 1."""
    rng = np.random.default_rng(n)
    pos = rng.standard_normal((n, 3))
    mass = 2.0 ** -136 * (np.ones(n) if equal else rng.integers(1, 3, n))
    with nb.Simulation(n, "mixed", eps=0.5) as sim:
        acc, pot = sim.accel(pos, mass)
    oa, op, _ = oracle.accel(pos, mass, 0.5)
    assert 1e-40 < np.abs(oa).max() < 2.0 ** -126
    assert (np.abs(acc - oa) <= 4 * n * 2.0 ** -150 + 1e-5 * np.abs(oa).max()).all()
    assert (np.abs(pot - op) <= 4 * n * 2.0 ** -150 + 1e-5 * np.abs(op)).all()


@pytest.mark.parametrize("n", [25, 300, 1200])
@pytest.mark.parametrize("sym", [0, 1])
def test_f64e_small_masses(nb, n, sym):
    """Sums near and below binary32's normal numbers: m / r^3 >= 2.6e-38 is off by up to
    2^-149 in each of its two products and its low part, which is what bounds the forces."""
    rng = np.random.default_rng(n)
    pos = 10.0 * rng.standard_normal((n, 3))
    mass = np.full(n, 4e-32)
    with nb.Simulation(n, "f64e", eps=100.0) as sim:
        sim.set_symmetric(sym)
        acc, pot = sim.accel(pos, mass)
    oa, op, smag = oracle.accel(pos, mass, 100.0)
    assert (np.linalg.norm(acc - oa, axis=1) <= 3 * 2.0 ** -149 / 2.6e-38 * smag).all()
    assert (np.abs(pot - op) <= 1e-12 * np.abs(op)).all()
