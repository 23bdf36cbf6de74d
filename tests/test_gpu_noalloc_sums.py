"""Mean stress of hmc_stress_noalloc against the FP64 sum of the stress that it returns, per component,
where the terms of a sum cancel; on grids whose threads take one cell and four, with a last CTA that is
part-filled, on pointers that allow the wide accesses and on others that do not (the same bits).

Tolerance: a thread adds n terms (8 a cell) as a TwoSum pair of FP32 numbers, u = 2^-24.  Only the sum of the
error terms is rounded: n additions of at most n u sum|x| each, then ten more over the warp, which is below
(n + 10)^2 u^2 of the sum of the terms' magnitudes; the FP64 sums above add less than 2^-45 of it.  A sum
whose additions lose bits (about u sqrt(threads) of the terms) lies far outside."""
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


# 60 and 448 cells: one cell a thread; 90 945 cells, 356 CTAs of which the last has 65: four
@pytest.mark.parametrize("shape,cells", [((6, 10, 8), 1), ((14, 16, 16), 1), ((86, 90, 94), 4)])
def test_mean_of_cancelling_terms(G, shape, cells):
    import torch
    Q, (nz, ny, nx) = 7, shape
    spins = S.random_spins(shape, Q, 4)
    spins[: nz // 2] = spins[0, 0, 0]        # half the cells keep one orientation
    rng = np.random.default_rng(5)
    u = (rng.standard_normal((spins.size // 8, 3)) * 1e-3).astype(np.float32)
    C = O.tables(S.euler_uniform_so3(Q, 3), **C3)[1].astype(np.float32)
    got = []
    for off in ((0, 0, 0, 0), (2, 4, 4, 4), (0, 0, 0, 8)):   # spins, u, ctab, sigma
        keep = [_at(torch, a, o) for a, o in zip((spins, u, C, np.zeros(spins.size * 6, np.float32)), off)]
        mean = torch.zeros(6, dtype=torch.float64, device="cuda:0")
        energy = torch.zeros(1, dtype=torch.float64, device="cuda:0")
        torch.cuda.synchronize()
        s, du, c, sig = (v.data_ptr() for _, v in keep)
        G.hmc_stress_noalloc(s, du, c, np.zeros(6), nx, ny, nz, sig, mean.data_ptr(), energy.data_ptr(), None)
        torch.cuda.synchronize()
        got.append((keep[3][1].cpu().numpy().view(np.float32).reshape(-1, 6), mean.cpu().numpy(), energy.item()))
        assert not keep[3][0].cpu().numpy()[off[3] + 24 * spins.size:].any()    # nothing past its end
    sig, mean, energy = got[0]
    ref, size = sig.astype(np.float64).sum(0), np.abs(sig.astype(np.float64)).sum(0)
    tol = (8 * cells + 10) ** 2 * 2.0 ** -48 + 2.0 ** -45
    err = np.abs(mean * spins.size - ref) / size
    assert (err <= tol).all(), (err, tol)
    # the stored stress itself: FP32 rounding of the gradients and the Hooke products
    e = np.zeros(6)
    g = G.HMC(shape, Q, precision=G.HMC_FP32, bc=G.HMC_BC_STRAIN6, strain6=e, mpm_steps_per_mcs=0, **C3)
    g.set_orientations(S.euler_uniform_so3(Q, 3), spins)
    g.set_nodal(u.astype(np.float64), np.zeros(u.shape))
    g.compute_stress()
    assert np.linalg.norm(sig - g.stress()) < 2e-6 * np.linalg.norm(sig)
    g.close()
    for other in got[1:]:
        assert np.array_equal(other[0], sig) and np.array_equal(other[1], mean) and other[2] == energy
