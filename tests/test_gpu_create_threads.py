"""Creating handles on one thread leaves the launches of another alone: the kernels' shared-memory
limits are process-wide, and no creation lowers one that another handle's launches need (512
orientations: a table of 24 KB behind the tiles of a march)."""
import threading

import pytest

import hmc_synth as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    from conftest import build_libhmc
    build_libhmc()
    import paper_1009_0457_gb300 as G
    return G


def test_launches_beside_creations(G, monkeypatch):
    monkeypatch.setenv("HMC_MPM_SHAPE", "7")      # four marches to a CTA: more than the default limit of 48 KB
    shape, Q = (16, 16, 16), 512
    g = G.HMC(shape, Q, precision=G.HMC_FP32)
    g.set_orientations(S.euler_uniform_so3(Q, 2), S.random_spins(shape, Q, 3))
    g.mpm_steps(2)
    done, errors, rounds = threading.Event(), [], [0]

    def launch():
        while not done.is_set() and not errors:
            try:
                g.mpm_steps(2000)
                rounds[0] += 1
            except G.HMCError as e:
                errors.append(str(e))

    t = threading.Thread(target=launch)
    t.start()
    try:
        for _ in range(60):
            G.HMC((8, 8, 8), 4, precision=G.HMC_FP32).close()
    finally:
        done.set()
        t.join()
    g.synchronize()
    g.close()
    assert not errors and rounds[0] > 0
