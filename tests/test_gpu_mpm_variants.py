"""Every decomposition of the MPM step gives the same bits: marches over patches of any size,
one-pass blocks, on grids of one cell per edge upwards, thin and ragged ones, and batches
whose replicas are divided differently."""
import numpy as np
import pytest

import hmc_synth as S

pytestmark = pytest.mark.gpu

C3 = dict(c11=246.5, c12=147.3, c44=124.7)
VARIANTS = {0: "0123456", 1: "0123456789"}   # by precision


@pytest.fixture(scope="module")
def G():
    from conftest import build_libhmc
    build_libhmc()
    import paper_1009_0457_gb300 as G
    return G


def _field(shape, Q, seed):
    return S.voronoi_spins(shape, max(2, int(np.prod(shape)) // 150), Q, seed)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("shape", [(4, 4, 4), (4, 4, 200), (120, 4, 6), (6, 90, 4), (16, 18, 20), (34, 62, 66)])
def test_variants_are_bitwise_equal(G, monkeypatch, shape, precision):
    Q = 300 if precision else 9     # FP32: above the block form's staged table
    eul, sp = S.euler_uniform_so3(Q, 2), _field(shape, Q, 4)
    u0 = np.random.default_rng(3).normal(size=(np.prod(shape) // 8, 3)) * 1e-3
    out = []
    for v in VARIANTS[precision]:
        monkeypatch.setenv("HMC_MPM_SHAPE", v)
        g = G.HMC(shape, Q, precision=precision, load_axis=(1, 2, 3.0), strain=2e-3, **C3)
        g.set_orientations(eul, sp)
        g.set_nodal(u0, None)
        g.mpm_steps(3)
        assert g.tuning()[0] == int(v)
        out.append(g.nodal())
        g.close()
    assert np.isfinite(out[0][0]).all() and np.abs(out[0][1]).max() > 0
    for u, v in out[1:]:
        assert np.array_equal(u, out[0][0]) and np.array_equal(v, out[0][1])


@pytest.mark.parametrize("precision", [0, 1])
def test_batch_variants_equal_solo_runs(G, monkeypatch, precision):
    Q, shapes = 9, [(4, 4, 4), (32, 32, 32), (10, 50, 100)]
    eul = S.euler_uniform_so3(Q, 2)
    fields = [_field(s, Q, 7 + i) for i, s in enumerate(shapes)]
    common = dict(precision=precision, strain=2e-3, **C3)
    monkeypatch.setenv("HMC_MPM_SHAPE", "0")
    ref = []
    for s, f in zip(shapes, fields):
        g = G.HMC(s, Q, **common)
        g.set_orientations(eul, f)
        g.mpm_steps(4)
        ref.append(g.nodal()[0])
        g.close()
    for v in VARIANTS[precision]:
        monkeypatch.setenv("HMC_MPM_SHAPE", v)
        b = G.HMCBatch(shapes, Q, **common)
        b.set_orientations(eul, fields)
        b.mpm_steps(4)
        for r in range(len(shapes)):
            assert np.array_equal(b.nodal(r)[0], ref[r]), (v, r)
        b.close()
