"""Zone half sweeps whose trials are decided by bounds, by the elimination, or both: FP64 decisions
identical to the oracle's zone re-solve from weak to overwhelming elastic energy (few to most trials
left open), at kT = 0, and for a nearly singular stiffness, where the bounds are not used.  At kT = 0
the threshold is zero, and a trial between equal orientations and equal neighbourhoods is a tie there:
the library has dH = 0 exactly, the oracle's re-solve 1e-13 of either sign, so a decision may differ
where |dH - t| <= 1e-9 max(1, |t|), the criterion of the zone's other FP64 parity tests."""
import numpy as np
import pytest

import hmc_synth as S
import oracle as O
import oracle.zone as Z

pytestmark = pytest.mark.gpu

NI, THIN = (246.5, 147.3, 124.7), (100.0, 10.0, 3000.0)
EB = np.array([-7e-4, -6e-4, 2e-3, 2e-4, -4e-4, 1e-4])


@pytest.fixture(scope="module")
def G():
    from conftest import build_libhmc
    build_libhmc()
    import paper_1009_0457_gb300 as G
    return G


@pytest.mark.parametrize("c,lam,kT", [(NI, 30.0, 0.7), (NI, 2e3, 0.7), (NI, 2e4, 0.7), (NI, 3e6, 0.7), (NI, 2e4, 0.0),
                                      (THIN, 2e3, 0.7)])
def test_decisions_equal_the_oracles(G, c, lam, kT):
    shape, Q, seed = (8, 6, 10), 7, 21
    kw = dict(zip(("c11", "c12", "c44"), c))
    eul, sp = S.euler_uniform_so3(Q, 4), S.random_spins(shape, Q, 5)
    eul[2] = eul[1]                       # trials between equal orientations fall to the Potts rule
    _, Ct, _ = O.tables(eul, **kw)
    u = np.random.default_rng(6).normal(size=(sp.size // 8, 3)) * 1e-3
    g = G.HMC(shape, Q, precision=G.HMC_FP64, elastic=G.HMC_ELASTIC_ZONE1, elastic_scale=lam, kT=kT, bc=G.HMC_BC_STRAIN6,
              strain6=tuple(EB), mpm_steps_per_mcs=0, seed=seed, **kw)
    g.set_orientations(eul, sp)
    g.set_nodal(u, np.zeros_like(u))
    Bs = Z.all_strain_matrices(shape)
    spo, total = sp.copy(), 0
    for colour in (0, 1):
        acc = g.sweep_half(colour)
        acc_o, _, dH, t = Z.half_sweep_zone(spo, colour, seed, 0, 0, 1.0, kT, 0, Q, lam, Ct, EB, u.reshape(-1), 1, Bs)
        differ = np.flatnonzero((g.spins() != spo).ravel())
        assert (np.abs(dH - t)[differ] <= 1e-9 * np.maximum(1.0, np.abs(t[differ]))).all()
        assert abs(acc - acc_o) <= len(differ) and (kT == 0.0 or len(differ) == 0)
        g.set_spins(spo)
        total += acc
    assert total > 0 and g.info().zone_trials > 50
    g.close()
