"""A handle that is given new orientations after it has run, FP64: the fixed-point stiffness table
takes another exponent where the largest row sum passes a power of two (iron: 501 GPa aligned,
562 to 569 turned), and every launch that follows uses it, those of graphs captured before included:
the same bits as a fresh handle."""
import numpy as np
import pytest

import hmc_synth as S

pytestmark = pytest.mark.gpu

IRON = dict(c11=231.4, c12=134.7, c44=116.4)
SHAPE, Q = (12, 14, 20), 6
SETS = {"aligned": np.zeros((Q, 3)), "turned": S.euler_uniform_so3(Q, 2)}


@pytest.fixture(scope="module")
def G():
    from conftest import build_libhmc
    build_libhmc()
    import paper_1009_0457_gb300 as G
    return G


def _state(g):
    return g.strain(), g.spins(), *g.nodal()


@pytest.mark.parametrize("mpm", [3, 10])       # eight steps and one step to a graph
@pytest.mark.parametrize("order", [("aligned", "turned"), ("turned", "aligned")])
def test_steps_after_new_orientations_equal_a_fresh_handle(G, order, mpm):
    sp = S.voronoi_spins(SHAPE, 30, Q, 2)
    out = []
    for names in (order, order[1:]):
        g = G.HMC(SHAPE, Q, precision=G.HMC_FP64, strain=2e-3, mpm_steps_per_mcs=mpm, seed=3, **IRON)
        for name in names:
            g.set_orientations(SETS[name], sp)
            g.mc_sweeps(17)
        out.append(_state(g))
        g.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("order", [("aligned", "turned"), ("turned", "aligned")])
def test_a_callers_graph_of_steps_follows_new_orientations(G, order):
    import torch
    sp = S.voronoi_spins(SHAPE, 30, Q, 2)
    s = torch.cuda.Stream()
    out = []
    for names in (order, order[1:]):
        g = G.HMC(SHAPE, Q, precision=G.HMC_FP64, strain=2e-3, stream=s.cuda_stream, **IRON)
        g.set_orientations(SETS[names[0]], sp)
        if len(names) == 2:
            g.mpm_steps(2)
            with torch.cuda.stream(s):
                graph = torch.cuda.CUDAGraph()
                graph.capture_begin()
                g.mpm_steps(2)
                graph.capture_end()
                g.set_orientations(SETS[names[1]], sp)
                graph.replay()
        else:
            g.mpm_steps(2)
        g.synchronize()
        out.append(_state(g))
        g.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
