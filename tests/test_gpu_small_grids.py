"""The forms that small grids take: the stress pass with one block per thread gives the bits of the
other form (a batch large enough for the other form equals the solo runs), the end-of-step
reduction with one and with several CTAs per replica agrees with the oracle's means, and the
grain count by block labels equals a flood fill on grids two blocks wide and on checkered ones;
steps run several to a graph equal single steps."""
import numpy as np
import pytest

import hmc_synth as S
import oracle as O

pytestmark = pytest.mark.gpu

C3 = dict(c11=246.5, c12=147.3, c44=124.7)


@pytest.fixture(scope="module")
def G():
    from conftest import build_libhmc
    build_libhmc()
    import paper_1009_0457_gb300 as G
    return G


@pytest.mark.parametrize("precision", [0, 1])
def test_stress_forms_give_the_same_bits(G, precision):
    # 20 replicas of 25 to 26 tiles: above the wide form's line in FP32 and FP64, each below it alone
    Q, shapes = 9, [(30, 36, 48)] * 19 + [(34, 38, 40)]
    eul = S.euler_uniform_so3(Q, 2)
    fields = [S.voronoi_spins(s, 60, Q, 3) for s in shapes[-2:]]
    fields = [fields[0]] * 19 + [fields[1]]
    common = dict(precision=precision, strain=2e-3, mpm_steps_per_mcs=3, **C3)
    b = G.HMCBatch(shapes, Q, [dict(seed=5)] * 20, **common)
    b.set_orientations(eul, fields)
    b.mc_sweeps(2)
    for r in (0, 19):
        g = G.HMC(shapes[r], Q, seed=5, **common)
        g.set_orientations(eul, fields[r])
        g.mc_sweeps(2)
        assert np.array_equal(g.strain(), b.strain(r)) and np.array_equal(g.spins(), b.spins(r))
        assert np.array_equal(g.nodal()[1], b.nodal(r)[1])
        g.close()
    b.close()


# one CTA per replica up to 512 stress CTAs (2^17 blocks), several above
@pytest.mark.parametrize("shape", [(4, 4, 4), (6, 10, 34), (64, 128, 128), (66, 128, 128)])
def test_mean_stress_and_energy_equal_the_sums_of_the_stored_stress(G, shape):
    Q = 7
    g = G.HMC(shape, Q, precision=G.HMC_FP64, strain=2e-3, mpm_steps_per_mcs=0, **C3)
    sp = S.box_grain_spins(shape, 5, Q, 3)
    g.set_orientations(S.euler_uniform_so3(Q, 2), sp)
    g.mpm_steps(2)
    mean, energy = g.compute_stress()
    sig, n = g.stress(), sp.size
    S6 = O.tables(S.euler_uniform_so3(Q, 2), **C3)[2][sp.ravel()]
    g.close()
    # sums of n values in another order: n/2 roundings of 2^-53 on average cancel to sqrt(n)
    assert np.abs(mean - sig.mean(0)).max() <= 1e-12 * np.abs(sig).max()
    assert abs(energy - 0.5 * np.einsum("ni,nij,nj->", sig, S6, sig)) <= 1e-11 * abs(energy)


@pytest.mark.parametrize("shape,Q", [((4, 4, 4), 2), ((4, 4, 40), 3), ((6, 30, 4), 2), ((20, 22, 26), 4)])
@pytest.mark.parametrize("kind", ["random", "voronoi", "checkered", "one"])
def test_grain_count_by_block_labels(G, shape, Q, kind):
    z, y, x = np.indices(shape)
    sp = {"random": S.random_spins(shape, Q, 3), "voronoi": S.voronoi_spins(shape, 9, Q, 3),
          "checkered": ((x + y + z) % 2).astype(np.uint16), "one": np.zeros(shape, np.uint16)}[kind]
    g = G.HMC(shape, Q, elastic=0, mpm_steps_per_mcs=0)
    g.set_orientations(S.euler_uniform_so3(Q, 2), sp)
    n = g.grain_count()
    g.close()
    assert n == O.grain_count(sp)


# steps of at most eight launches run in graphs of eight steps, the rest of them one by one: equal to
# single steps for counts around the multiples, with an even and an odd number of MPM steps
@pytest.mark.parametrize("mpm", [0, 1, 3, 4, 5])
def test_many_steps_equal_single_steps(G, mpm):
    shape, Q = (12, 14, 10), 9
    eul, sp = S.euler_uniform_so3(Q, 2), S.voronoi_spins(shape, 40, Q, 3)
    out = []
    for counts in ([1] * 35, [7, 8, 19, 1], [35]):
        g = G.HMC(shape, Q, precision=1, strain=2e-3, mpm_steps_per_mcs=mpm, seed=5, **C3)
        g.set_orientations(eul, sp)
        acc = sum(g.mc_sweeps(n) for n in counts)
        out.append((acc, g.spins(), g.strain(), *g.nodal()))
        g.close()
    for other in out[1:]:
        for a, b in zip(out[0], other):
            assert np.array_equal(a, b)


def test_fp64_stress_forms_on_both_sides_of_the_line(G):
    # 56, 59 and 61 tiles: alone the first is spread over clusters and the others take one CTA a tile; all
    # three together (176) take the form of large grids
    Q, shapes = 9, [(44, 52, 50), (46, 52, 50), (48, 52, 50)]
    eul = S.euler_uniform_so3(Q, 2)
    fields = [S.voronoi_spins(s, 60, Q, 3) for s in shapes]
    common = dict(precision=0, strain=2e-3, mpm_steps_per_mcs=2, **C3)
    b = G.HMCBatch(shapes, Q, [dict(seed=5)] * 3, **common)
    b.set_orientations(eul, fields)
    b.mc_sweeps(2)
    for r, shape in enumerate(shapes):
        g = G.HMC(shape, Q, seed=5, **common)
        g.set_orientations(eul, fields[r])
        g.mc_sweeps(2)
        assert np.array_equal(g.strain(), b.strain(r)) and np.array_equal(g.spins(), b.spins(r))
        assert np.array_equal(g.nodal()[1], b.nodal(r)[1])
        g.close()
    b.close()
