"""One FP64 MPM step from rest, component by component, on states whose components differ: a common
displacement along one axis (large against the strains, also against everything a cell's exponent could
take in) leaves the forces of all three axes as accurate as without it, and a component that is small
everywhere is wrong by no more than the bound that holds for the largest.

Tolerance: a step rounds each strain and each stress component of a point at 2^-52 or better of the largest
of its cell, and a node's force sums at most 64 of them: 64 x 2^-52 = 1.4e-14 of the largest component's norm, and the
oracle's FP64 sums carry as much: 3e-14.  (Aligned to the largest displacement of a cell instead, an offset of
1e3 beside 1e-3 cost 1e-11.)"""
import numpy as np
import pytest

import hmc_synth as S
import oracle as O

pytestmark = pytest.mark.gpu

EB = (-7e-4, -6e-4, 2e-3, 2e-4, -4e-4, 1e-4)
C3 = dict(c11=246.5, c12=147.3, c44=124.7)


@pytest.fixture(scope="module")
def G():
    from conftest import build_libhmc
    build_libhmc()
    import paper_1009_0457_gb300 as G
    return G


def _step(G, shape, eul, sp, u0, eb, variant, monkeypatch, offset=0.0):
    """The velocity after one step of the library, and the oracle's from the state without the offset, which
    exerts no force (the oracle sums shape-function gradients times displacements, not differences of
    displacements, so it would carry 2^-53 of the offset itself; subtracting it is exact)."""
    monkeypatch.setenv("HMC_MPM_SHAPE", variant)
    g = G.HMC(shape, len(eul), precision=G.HMC_FP64, bc=G.HMC_BC_STRAIN6, strain6=eb, **C3)
    g.set_orientations(eul, sp)
    g.set_nodal(u0, np.zeros_like(u0))
    g.mpm_steps(1)
    v = g.nodal()[1]
    g.close()
    vo, uo = np.zeros_like(u0), u0 - offset
    O.mpm_steps(sp, O.tables(eul, **C3)[1], np.array(eb), uo, vo, 1, O.default_dt(**C3), 0.05)
    return v, vo


@pytest.mark.parametrize("variant", ["0", "5", "6"])     # march, blocks of whole cells and of quarters
@pytest.mark.parametrize("eb", [EB, (0.0,) * 6])
@pytest.mark.parametrize("offset", [(0, 0, 0), (50, 0, 0), (0, -1e3, 0), (0, 0, 3e7), (1e9, 0, -20), (0.5, 0.5, -0.5)])
def test_an_offset_along_an_axis_costs_no_accuracy(G, offset, eb, variant, monkeypatch):
    shape, Q = (10, 38, 36), 9
    eul, sp = S.euler_uniform_so3(Q, 2), S.voronoi_spins(shape, 30, Q, 2)
    u0 = 1e-3 * np.random.default_rng(3).normal(size=(sp.size // 8, 3)) + np.array(offset, float)
    v, vo = _step(G, shape, eul, sp, u0, eb, variant, monkeypatch, np.array(offset, float))
    for d in range(3):
        assert np.linalg.norm(v[:, d] - vo[:, d]) <= 3e-14 * np.linalg.norm(vo, axis=0).max(), d


@pytest.mark.parametrize("variant", ["0", "5", "6"])
@pytest.mark.parametrize("small", [1e-3, 1e-9])
def test_a_small_component_is_held_to_the_largest(G, small, variant, monkeypatch):
    # aligned crystals, a transverse wave beside a longitudinal one along x: the components decouple
    shape, Q = (10, 38, 36), 2
    sp = S.voronoi_spins(shape, 30, Q, 2)
    x = np.arange(sp.size // 8) % (shape[2] // 2)
    w = 1e-3 * np.sin(2 * np.pi * x / (shape[2] // 2))
    u0 = np.stack([w, small * w, 0 * w], axis=1)
    v, vo = _step(G, shape, np.zeros((Q, 3)), sp, u0, (0.0,) * 6, variant, monkeypatch)
    for d in range(3):
        assert np.linalg.norm(v[:, d] - vo[:, d]) <= 3e-14 * np.linalg.norm(vo[:, 0]), d


def test_subnormal_displacements_exert_forces(G, monkeypatch):
    # 1e-310 has 44 bits; the sums of either form round at 2^-1074, at most a few thousand times (64 products
    # with a stiffness of some hundreds): 1e-320, beside the 3e-14 of the values
    shape, Q = (10, 12, 14), 5
    eul, sp = S.euler_uniform_so3(Q, 2), S.voronoi_spins(shape, 30, Q, 2)
    u0 = 1e-310 * np.random.default_rng(3).normal(size=(sp.size // 8, 3))
    for variant in "056":
        v, vo = _step(G, shape, eul, sp, u0, (0.0,) * 6, variant, monkeypatch)
        assert np.abs(vo).max() > 1e-310 and np.abs(v - vo).max() <= 3e-14 * np.abs(vo).max() + 1e-320
