"""hmc_mc_sweeps while a caller captures work of its own on another stream: a first call on each
displacement buffer, with any number of steps, is all that has to come before the capture (the
library's own graphs are of one step and of eight; neither disturbs the capture)."""
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


@pytest.mark.parametrize("first", [1, 8])
@pytest.mark.parametrize("mpm", [0, 1, 2, 10])
def test_steps_beside_a_callers_capture(G, mpm, first):
    import torch
    shape, Q, n = (12, 14, 20), 9, 18
    eul, sp = S.euler_uniform_so3(Q, 2), S.voronoi_spins(shape, 30, Q, 2)
    x = torch.zeros(1000, device="cuda:0")
    torch.cuda.synchronize()
    out = []
    for capture in (True, False):
        g = G.HMC(shape, Q, precision=G.HMC_FP32, strain=2e-3, mpm_steps_per_mcs=mpm, seed=3)
        g.set_orientations(eul, sp)
        if capture:
            G.hmc_mc_sweeps(g.h, first, want_accepted=False)
            G.hmc_mc_sweeps(g.h, 1, want_accepted=False)
            g.synchronize()
            graph, error = torch.cuda.CUDAGraph(), None
            with torch.cuda.stream(torch.cuda.Stream()):
                graph.capture_begin()
                x.add_(1)
                try:
                    G.hmc_mc_sweeps(g.h, n, want_accepted=False)
                except G.HMCError as e:
                    error = e
                graph.capture_end()
                graph.replay()
            torch.cuda.synchronize()
            assert error is None and (x == 1).all()
        else:
            g.mc_sweeps(first + 1 + n)
        g.synchronize()
        out.append((g.strain(), g.spins(), *g.nodal()))
        g.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
