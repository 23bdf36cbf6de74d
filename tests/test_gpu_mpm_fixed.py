"""The FP64 MPM step runs in 64-bit fixed point with one exponent per cell: it agrees
with the FP64 oracle over nodal states whose magnitudes differ by many orders within a
cell, between cells and against the mean strain, whatever the unit of the stiffness.

Tolerance: a stress component is rounded once, at 2^-50 or better of the largest stress of
its cell, and a displacement once at 2^-53 of the largest of its cell; the forces are sums
of at most 64 of them, so a step's relative error (2-norm) stays below 64 x 2^-50 = 6e-14,
and that of ``STEPS`` steps below 1e-12.
"""
import numpy as np
import pytest

import hmc_synth as S
import oracle as O

pytestmark = pytest.mark.gpu

STEPS = 6
EB = (-7e-4, -6e-4, 2e-3, 2e-4, -4e-4, 1e-4)


@pytest.fixture(scope="module")
def G():
    from conftest import build_libhmc
    build_libhmc()
    import paper_1009_0457_gb300 as G
    return G


def _rel(a, b):
    m = np.abs(b).max()      # squares of the tiny state would underflow
    return np.linalg.norm((a - b) / m) / np.linalg.norm(b / m)


def _state(kind, n, rng):
    """(u, v, mean strain) of n nodes."""
    u, v = rng.normal(size=(n, 3)), rng.normal(size=(n, 3)) * 1e-2
    if kind == "usual":
        return 1e-3 * u, 1e-3 * v, EB
    if kind == "rough":          # displacements far above the mean strain
        return 1e3 * u, 1e3 * v, EB
    if kind == "unstrained":
        return u, v, (0.0,) * 6
    if kind == "tiny":           # far below every exponent that a scale factor could take up
        return 1e-280 * u, 1e-280 * v, (0.0,) * 6
    if kind == "spread":         # twelve orders of magnitude between nodes
        return u * 10.0 ** rng.uniform(-12, 0, size=(n, 1)), 0 * v, tuple(1e-6 * x for x in EB)
    if kind == "one_node":
        w = 0 * u
        w[n // 3] = (1e-3, 0.0, -2e-7)
        return w, 0 * v, (0.0,) * 6
    if kind == "drift":          # a common displacement much larger than its differences
        return 50.0 + 1e-3 * u, 0 * v, EB
    raise ValueError(kind)


@pytest.mark.parametrize("scale", [1.0, 3e-7])
@pytest.mark.parametrize("kind", ["usual", "rough", "unstrained", "tiny", "spread", "one_node", "drift"])
def test_states_of_any_magnitude_match_the_oracle(G, kind, scale):
    shape, Q = (10, 38, 36), 9    # two tiles each way, the last one ragged
    rng = np.random.default_rng(3)
    eul = S.euler_uniform_so3(Q, 2)
    eul[0] = 0.0                  # an aligned crystal: exact zeros in its stiffness
    sp = S.voronoi_spins(shape, 30, Q, 2)
    u0, v0, eb = _state(kind, sp.size // 8, rng)
    c = dict(c11=246.5 * scale, c12=147.3 * scale, c44=124.7 * scale)
    dt = O.default_dt(**c)
    g = G.HMC(shape, Q, precision=G.HMC_FP64, bc=G.HMC_BC_STRAIN6, strain6=eb, **c)
    g.set_orientations(eul, sp)
    g.set_nodal(u0, v0)
    g.mpm_steps(STEPS)
    u, v = g.nodal()
    g.close()
    uo, vo = u0.copy(), v0.copy()
    O.mpm_steps(sp, O.tables(eul, **c)[1], np.array(eb), uo, vo, STEPS, dt, 0.05)
    # "drift": differences of the displacement carry an error of 2^-53 of it in either form
    tol = 1e-12 if kind != "drift" else 1e-12 * 50.0 / 1e-3
    assert _rel(u, uo) <= 1e-12
    assert _rel(v, vo) <= tol


def test_a_non_finite_displacement_reaches_its_neighbours_only(G, monkeypatch):
    shape, Q = (12, 12, 40), 4
    g = G.HMC(shape, Q, precision=G.HMC_FP64, bc=G.HMC_BC_STRAIN6, strain6=EB)
    g.set_orientations(S.euler_uniform_so3(Q, 2), S.voronoi_spins(shape, 20, Q, 2))
    monkeypatch.setenv("HMC_FAULT", "nan")      # a NaN in the first node's displacement
    with pytest.raises(G.HMCError):
        g.compute_stress()
    monkeypatch.delenv("HMC_FAULT")
    g.mpm_steps(1)
    v = g.nodal()[1].reshape(6, 6, 20, 3)
    g.close()
    near = np.zeros((6, 6, 20), dtype=bool)
    near[np.ix_((-1, 0, 1), (-1, 0, 1), (-1, 0, 1))] = True
    assert np.isnan(v[near]).all() and np.isfinite(v[~near]).all()
