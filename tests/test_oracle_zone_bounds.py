"""The two bounds of the 27-point zone's energy shift that decide most trials without a zone
solve hold against the oracle's zone re-solve: with R the resistance of the zone's other points to
a strain of its site, dH = 1/2 e0.w - 1/2 w.(C_new + R)^-1 w, and R lies between those of the two
isotropic surroundings with the crystal's bulk modulus and its smaller and larger shear modulus.
For strong and weak cubic anisotropy, any strain and neighbourhood, every position of the site
in its cell, and trials between equal orientations, where all are zero."""
import numpy as np
import pytest

import hmc_synth as S
import oracle as O
import oracle.zone as Z


def _resistance(par, C):
    """R of an isotropic zone C at a site of parities par."""
    shape = (8, 8, 8)
    x, y, z = (2 + p for p in par)
    Bs = [Z.strain_matrix(shape, x + dx, y + dy, z + dz) for dz in (-1, 0, 1) for dy in (-1, 0, 1) for dx in (-1, 0, 1)]
    K = sum(np.asarray(B).T @ C @ np.asarray(B) for B in Bs)
    Bp = np.asarray(Bs[13])
    on = np.flatnonzero(np.abs(K).sum(0) > 0)
    G = Bp[:, on] @ np.linalg.pinv(K[np.ix_(on, on)], rcond=1e-10, hermitian=True) @ Bp[:, on].T
    return np.linalg.inv(G) - C


def _isotropic(c11, c12, c44, pick):
    m2 = pick(c11 - c12, 2 * c44)
    C = np.zeros((6, 6))
    C[:3, :3] = (c11 + 2 * c12 - m2) / 3
    C[range(3), range(3)] += m2
    C[range(3, 6), range(3, 6)] = m2 / 2
    return C


@pytest.mark.parametrize("c", [(246.5, 147.3, 124.7), (246.5, 147.3, 49.6), (100.0, 10.0, 300.0), (300.0, 290.0, 80.0)])
def test_bounds_hold_for_the_zone_shift(c):
    rng = np.random.default_rng(17)
    shape, Q = (8, 10, 8), 5
    sp = rng.integers(0, Q, size=shape).astype(np.uint16)
    eul = S.euler_uniform_so3(Q, 3)
    eul[1] = eul[0]                       # two equal orientations
    _, Ct, _ = O.tables(eul, *c)
    E = rng.normal(size=6) * 1e-3
    u = rng.normal(size=(sp.size // 8, 3)) * 1e-3
    soft, stiff = _isotropic(*c, min), _isotropic(*c, max)
    for pos in range(8):
        par = (pos & 1, pos >> 1 & 1, pos >> 2)
        Rs, Rh = _resistance(par, soft), _resistance(par, stiff)
        for _ in range(15):
            x, y, z = (2 * int(rng.integers(0, n // 2)) + p for n, p in zip(shape[::-1], par))
            q, qn = int(sp[z, y, x]), int(rng.integers(0, Q))
            dH = Z.zone_shift_local(sp, Ct, E, u, x, y, z, qn)
            e0 = O.point_strain(shape, u, E, x, y, z)
            w = (Ct[qn] - Ct[q]) @ e0
            up = 0.5 * e0 @ w
            most, least = (0.5 * w @ np.linalg.solve(Ct[qn] + R, w) for R in (Rs, Rh))
            tol = 1e-8 * (abs(up) + most) + 1e-16      # rounding of the two solves
            assert 0 <= least <= most + tol
            assert up - most - tol <= dH <= up - least + tol, (pos, q, qn, dH, up, most, least)
