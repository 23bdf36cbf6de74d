"""hmc_stress_noalloc on grids whose cell rows are shorter and longer than a warp, filled and
part-filled CTAs, and on pointers that allow only the narrow accesses: the same bits whatever
the alignment, and the handle's own stress."""
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


def _at(torch, a, offset_bytes):
    """a on the device, `offset_bytes` past a 256-byte boundary."""
    raw = torch.zeros(a.nbytes + 512, dtype=torch.uint8, device="cuda:0")
    view = raw[offset_bytes:offset_bytes + a.nbytes]
    view.copy_(torch.from_numpy(a.reshape(-1).view(np.uint8).copy()))
    return raw, view


@pytest.mark.parametrize("shape", [(4, 4, 4), (4, 6, 66), (16, 16, 16), (10, 14, 38), (6, 4, 130), (34, 34, 16)])
def test_any_row_length_and_alignment(G, shape):
    import torch
    Q, (nz, ny, nx) = 7, shape
    eul = S.euler_uniform_so3(Q, 3)
    spins = S.random_spins(shape, Q, 4)
    spins[: nz // 2] = spins[0, 0, 0]        # half the cells keep one orientation
    rng = np.random.default_rng(5)
    u = (rng.standard_normal((spins.size // 8, 3)) * 1e-3).astype(np.float32)
    C = O.tables(eul, **C3)[1].astype(np.float32)
    g = G.HMC(shape, Q, precision=G.HMC_FP32, strain=2e-3, mpm_steps_per_mcs=0, **C3)
    g.set_orientations(eul, spins)
    g.set_nodal(u.astype(np.float64), np.zeros(u.shape))
    mean_ref, W_ref = g.compute_stress()
    sig_ref, E = g.stress(), g.strain()
    g.close()
    got = []
    for off in ((0, 0, 0, 0), (2, 4, 4, 4), (0, 0, 0, 8), (0, 0, 8, 0)):   # spins, u, ctab, sigma
        keep = [_at(torch, a, o) for a, o in zip((spins, u, C, np.zeros(spins.size * 6, np.float32)), off)]
        mean = torch.zeros(6, dtype=torch.float64, device="cuda:0")
        energy = torch.zeros(1, dtype=torch.float64, device="cuda:0")
        torch.cuda.synchronize()
        s, du, c, sig = (v.data_ptr() for _, v in keep)
        G.hmc_stress_noalloc(s, du, c, E, nx, ny, nz, sig, mean.data_ptr(), energy.data_ptr(), None)
        torch.cuda.synchronize()
        got.append((keep[3][1].cpu().numpy().view(np.float32), mean.cpu().numpy(), energy.item()))
        assert not keep[3][0].cpu().numpy()[off[3] + 24 * spins.size:].any()    # nothing past its end
    for sig, mean, energy in got:
        # 2e-6: FP32 rounding of the Hooke products, as the handle's own pass has it
        assert np.linalg.norm(sig.reshape(-1, 6) - sig_ref) < 2e-6 * np.linalg.norm(sig_ref)
        assert np.linalg.norm(mean - mean_ref) < 2e-6 * np.linalg.norm(mean_ref)
        assert abs(energy - W_ref) < 2e-6 * abs(W_ref)
        assert np.array_equal(sig, got[0][0]) and np.array_equal(mean, got[0][1]) and energy == got[0][2]
