"""Monte Carlo steps replayed from a graph, whose kernels start while the ones before them run,
equal the same phases called one by one with the device idle in between, bit for bit: the FP64
step in its block and march forms takes the mean strain of the end of the step before it, which
one CTA a replica forms, or several (above 512 stress tiles)."""
import numpy as np
import pytest

import hmc_synth as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    from conftest import build_libhmc
    build_libhmc()
    import paper_1009_0457_gb300 as G
    return G


@pytest.mark.parametrize("shapes,mpm,steps", [
    ([(12, 14, 10)], 1, 24),                       # eight steps to a graph
    ([(32, 32, 32)], 9, 6),
    ([(66, 128, 128), (16, 20, 18)], 2, 3),        # 528 stress tiles: more than one CTA at the end of a step
])
def test_overlapped_steps_equal_separate_phases(G, shapes, mpm, steps):
    Q = 9
    eul = S.euler_uniform_so3(Q, 2)
    fields = [S.box_grain_spins(s, 5, Q, 3) for s in shapes]
    out = []
    for graphs in (True, False):
        b = G.HMCBatch(shapes, Q, [dict(seed=5, replica=r) for r in range(len(shapes))], precision=G.HMC_FP64,
                       strain=2e-3, mpm_steps_per_mcs=mpm)
        b.set_orientations(eul, fields)
        if graphs:
            b.mc_sweeps(steps)
        else:
            for _ in range(steps):
                for phase in ([lambda: G.hmc_mpm_steps(b.h, 1)] * mpm +
                              [lambda: G.hmc_compute_stress(b.h), lambda: G.hmc_sweep_half(b.h, 0),
                               lambda: G.hmc_sweep_half(b.h, 1), lambda: G.hmc_end_mcs(b.h)]):
                    phase()
                    G.hmc_synchronize(b.h)
        out.append([x for r in range(len(shapes)) for x in (b.strain(r), b.spins(r), *b.nodal(r))])
        b.close()
    for a, c in zip(*out):
        assert np.array_equal(a, c)
