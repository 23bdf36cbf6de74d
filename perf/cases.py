"""The work that users of the hybrid Monte Carlo library have it do, as measurable cases.

Five kinds of call, each through the package's public functions:

* ``mc``: Monte Carlo steps of one replica.  A driver program holds the spin field on the
  GPU, hands it to the library, runs a few steps and takes the field back (zero copies to
  the host), as a loop around the library does between two of its own updates.
* ``batch``: one Monte Carlo step of an ensemble of replicas of uneven size.
* ``solve``: explicit MPM steps on a fixed microstructure from a given nodal state; the
  energy and the nodal fields come back to the host.
* ``stress``: the allocation-free stress pass on tensors of the caller.
* ``adjoint``: the elastic map with its gradient through ``HMCElastic``.

Handles compute in FP32 or FP64.  The C interface hands every number over as a double; what an
FP32 handle computed is returned as FP32 here, since that is all it holds.
"""
import math

import numpy as np
import torch

import paper_1009_0457_gb300 as G
from paper_1009_0457_gb300.autograd import HMCElastic

DEV = "cuda:0"
C11, C12, C44 = 246.5, 147.3, 124.7   # GPa, the nickel constants of the repository's workloads
VI, VJ = (0, 1, 2, 1, 0, 0), (0, 1, 2, 2, 2, 1)


def listed():
    mc = dict(kind="mc", elastic="traction", bc="uniaxial", trial="neighbor", strain=2e-3, kT=0.7, axis="z",
              grain=419, read="strain")
    return [
        # grain growth without load: the pure Potts field of the 60^3 growth study, its grains
        # counted every 25 steps; each step is a handful of small launches
        dict(mc, name="potts60", nx=60, ny=60, nz=60, Q=99, precision="fp32", elastic="off", mpm=0, mcs=25, kT=1.0,
             grain=1, read="grains"),
        # the 32^3 workload as configured: 10 steps of 50 MPM steps in FP64 (a study's reference run)
        dict(mc, name="ni32", nx=32, ny=32, nz=32, Q=64, precision="fp64", mpm=50, mcs=10, strain=1e-3, grain=164),
        # the same in the production precision: latency of small launches
        dict(mc, name="ni32_fp32", nx=32, ny=32, nz=32, Q=64, precision="fp32", mpm=50, mcs=10, strain=1e-3,
             grain=164),
        # the 128^3 workload, the ordinary size of a texture study
        dict(mc, name="ni128", nx=128, ny=128, nz=128, Q=256, precision="fp32", mpm=50, mcs=2),
        # the 256^3 workload (the repository's benchmark) with its texture log
        dict(mc, name="ni256", nx=256, ny=256, nz=256, Q=1024, precision="fp32", mpm=50, mcs=1, axis="111",
             read="texture"),
        # texture under tension: 100^3 (edges that no tile divides), 91 orientations about z, a load
        # ramp under stress control
        dict(mc, name="texture100", nx=100, ny=100, nz=100, Q=91, precision="fp32", bc="traction", mpm=50, mcs=4,
             kT=1.0, axis="x"),
        # the batched ensemble: replicas of the configured edges, one step of all of them
        dict(kind="batch", name="ensemble16", edges="48,64,96,128,160", replicas=16, Q=256, precision="fp32", mpm=50,
             mcs=1),
        # the 27-point zone at the size its workload is configured for
        dict(mc, name="zone128", nx=128, ny=128, nz=128, Q=256, precision="fp32", elastic="zone", mpm=50, mcs=1),
        # parameter gradients of the elastic solve, as configured: 200 steps, a checkpoint every 20
        dict(kind="adjoint", name="adjoint128", nx=128, ny=128, nz=128, Q=256, precision="fp32", steps=200,
             checkpoint=20, grain=419),
        # the stress pass inside another program's memory, at the largest cube it serves
        dict(kind="stress", name="stress256", nx=256, ny=256, nz=256, Q=1024, grain=419),
        # and on a small ragged box, where its launches are what it costs
        dict(kind="stress", name="stress_small", nx=38, ny=30, nz=34, Q=64, grain=164),
        # an elastic solve in FP64 with its fields read back: a reference solution
        dict(kind="solve", name="solve96_fp64", nx=96, ny=90, nz=100, Q=128, precision="fp64", steps=100, grain=419),
    ]


def draw(rng):
    def edges(lo, hi, most):
        # edges spread over their logarithm, even, any remainder of the tiles
        while True:
            e = [2 * int(round(math.exp(rng.uniform(math.log(lo / 2), math.log(hi / 2))))) for _ in range(3)]
            if rng.random() < 0.4:
                e = [e[0]] * 3
            if math.prod(e) <= most:
                return dict(nx=e[0], ny=e[1], nz=e[2])

    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["mc", "mc", "mc", "zone", "potts", "batch", "solve", "solve", "stress", "stress", "adjoint"])
    fp64 = rng.random() < 0.3
    prec = "fp64" if fp64 else "fp32"
    grain = log_int(100, 900)
    if kind in ("mc", "zone", "potts"):
        c = dict(kind="mc", elastic=rng.choice(["traction", "traction", "strain"]),
                 bc=rng.choice(["uniaxial", "uniaxial", "traction", "strain6"]),
                 trial=rng.choice(["neighbor", "neighbor", "uniform"]), strain=round(rng.uniform(5e-4, 3e-3), 5),
                 kT=rng.choice([0.7, 0.7, 1.0]), axis=rng.choice(["x", "z", "111"]), grain=grain,
                 read=rng.choice(["strain", "texture", "grains"]), Q=log_int(24, 2000), precision=prec,
                 mpm=rng.choice([20, 50, 51]), mcs=rng.choice([1, 2, 3]))
        if kind == "zone":
            c.update(elastic="zone", trial="neighbor", Q=log_int(24, 256), mcs=1)
        if kind == "potts":
            c.update(elastic="off", mpm=0, mcs=rng.choice([5, 20]))
        big = 1 << 24 if kind == "potts" else (1 << 16 if fp64 else 1 << 21) if kind == "zone" else \
            (1 << 20 if fp64 else 6 << 20)
        c.update(edges(16, 256, big))
        return c
    if kind == "batch":
        pool = sorted(rng.sample([16, 24, 32, 48, 50, 64, 80, 96, 128] if not fp64 else [16, 24, 32, 36, 48], 4))
        return dict(kind="batch", edges=",".join(map(str, pool)), replicas=rng.choice([4, 8, 13]), Q=log_int(32, 400),
                    precision=prec, mpm=rng.choice([20, 50]), mcs=1)
    if kind == "solve":
        c = dict(kind="solve", Q=log_int(24, 1500), precision=prec, steps=rng.choice([25, 60, 100]), grain=grain)
        c.update(edges(12, 160, 1 << 20))
        return c
    if kind == "stress":
        c = dict(kind="stress", Q=log_int(24, 2000), grain=grain)
        c.update(edges(12, 256, 1 << 24))
        return c
    c = dict(kind="adjoint", Q=log_int(24, 400), precision=prec, steps=rng.choice([20, 45, 80]),
             checkpoint=rng.choice([5, 10, 20]), grain=grain)
    c.update(edges(16, 128, 1 << 17 if fp64 else 1 << 20))
    return c


# ---- inputs -------------------------------------------------------------------

def _euler(Q, seed, about_z=False):
    """Q z-y-z Euler triples uniform on SO(3), or rotations about z by whole degrees."""
    if about_z:
        return np.stack([np.radians(np.arange(Q, dtype=float)), np.zeros(Q), np.zeros(Q)], axis=1)
    u = np.random.default_rng([seed, 1]).random((Q, 3))
    return np.stack([2 * np.pi * u[:, 0], np.arccos(1 - 2 * u[:, 1]), 2 * np.pi * u[:, 2]], axis=1)


def _polycrystal(nx, ny, nz, Q, grain, seed):
    """Orientation field (nz, ny, nx), int16: a periodic Voronoi polycrystal of about ``grain``
    voxels a grain (nearest seeds by jump flooding), or independent random orientations."""
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    if grain <= 1:
        return torch.randint(0, Q, (nz, ny, nx), generator=g, device=DEV, dtype=torch.int16)
    n = max(2, round(nx * ny * nz / grain))
    dims = (nz, ny, nx)
    box = torch.tensor([nz, ny, nx], device=DEV, dtype=torch.float32)
    pos = torch.rand(n, 3, generator=g, device=DEV) * box
    ori = torch.randint(0, Q, (n,), generator=g, device=DEV, dtype=torch.int16)
    cell = torch.minimum(pos.long(), (box - 1).long())
    flat = torch.full((nz * ny * nx,), -1, device=DEV, dtype=torch.int32)
    at = (cell[:, 0] * ny + cell[:, 1]) * nx + cell[:, 2]
    flat.scatter_reduce_(0, at, torch.arange(n, device=DEV, dtype=torch.int32), "amax")   # one seed a voxel
    own = flat.view(dims)
    axes = [torch.arange(m, device=DEV, dtype=torch.float32) + 0.5 for m in dims]

    def dist2(idx):
        d2 = None
        p = pos[idx.clamp_min(0).long()]
        for a in range(3):
            x = axes[a].view([-1 if b == a else 1 for b in range(3)])
            d = (p[..., a] - x).abs_()
            d = torch.minimum(d, box[a] - d).square_()
            d2 = d if d2 is None else d2.add_(d)
        return torch.where(idx < 0, torch.inf, d2)

    best = dist2(own)
    step = min(32, 1 << max(0, (round(2 * grain ** (1 / 3)) - 1).bit_length()))   # no seed is farther by much
    while step >= 1:
        for a in range(3):          # one axis after the other: the 27 neighbours of a step in three passes
            cand = [torch.roll(own, s, a) for s in (step, -step)]
            for c in cand:
                d = dist2(c)
                near = d < best
                own = torch.where(near, c, own)
                best = torch.where(near, d, best)
        step //= 2
    return ori[own.clamp_min(0).long()].contiguous()


def _params(c, seed):
    axis = dict(x=(1.0, 0.0, 0.0), z=(0.0, 0.0, 1.0))
    axis["111"] = (1.0, 1.0, 1.0)
    p = dict(c11=C11, c12=C12, c44=C44, kT=c["kT"], mpm_steps_per_mcs=c["mpm"], seed=int(seed) + 1,
             load_axis=axis[c["axis"]], strain=c["strain"],
             precision=G.HMC_FP64 if c["precision"] == "fp64" else G.HMC_FP32,
             elastic=dict(off=G.HMC_ELASTIC_OFF, traction=G.HMC_ELASTIC_TRACTION, zone=G.HMC_ELASTIC_ZONE1,
                          strain=G.HMC_ELASTIC_STRAIN)[c["elastic"]],
             trial=G.HMC_TRIAL_UNIFORM_Q if c["trial"] == "uniform" else G.HMC_TRIAL_NEIGHBOR,
             bc=dict(uniaxial=G.HMC_BC_UNIAXIAL, traction=G.HMC_BC_TRACTION, strain6=G.HMC_BC_STRAIN6)[c["bc"]])
    if c["bc"] == "strain6":
        p["strain6"] = tuple(x * c["strain"] for x in (-0.36, -0.31, 1.0, 0.1, -0.2, 0.05))
    if c["bc"] == "traction":
        p["stress"] = 0.0
    return p


def _prepare_mc(c, seed):
    spins = _polycrystal(c["nx"], c["ny"], c["nz"], c["Q"], c["grain"], seed)
    h = G.HMC((c["nz"], c["ny"], c["nx"]), c["Q"], **_params(c, seed))
    torch.cuda.synchronize()
    G.hmc_set_orientations_dev(h.h, _euler(c["Q"], seed, c["bc"] == "traction"), spins.data_ptr())
    ramp = [0.03 * (k + 1) / c["mcs"] for k in range(c["mcs"])] if c["bc"] == "traction" else None
    return dict(case=c, h=h, spins=spins, out=torch.empty_like(spins), ramp=ramp)


def _run_mc(s):
    c, h = s["case"], s["h"]
    G.hmc_set_spins_dev(h.h, s["spins"].data_ptr())
    accepted = 0
    if s["ramp"]:
        for load in s["ramp"]:
            h.set_load(load)
            accepted += h.mc_sweeps(1)
    else:
        accepted = h.mc_sweeps(c["mcs"])
    G.hmc_get_spins_dev(h.h, s["out"].data_ptr())
    r = dict(spins=s["out"], accepted=accepted)
    strain = h.strain()
    r["strain"] = strain if c["precision"] == "fp64" else strain.astype(np.float32)
    if c["read"] == "texture":
        r["fractions"], r["volumes"] = h.texture_histogram(G.HMC_HIST_ANGLE_100, 9)
    if c["read"] == "grains":
        r["grains"] = h.grain_count()
    return r


def _prepare_batch(c, seed):
    rng = np.random.default_rng([seed, 4])
    pool = [int(x) for x in c["edges"].split(",")]
    shapes, per, fields = [], [], []
    for r in range(c["replicas"]):
        e = pool[r % len(pool)]     # every edge in every ensemble, so that the work does not hang on the seed
        ax = rng.normal(size=3)
        shapes.append((e, e, e))
        per.append(dict(load_axis=tuple(ax / np.linalg.norm(ax)), strain=float(rng.uniform(5e-4, 3e-3)),
                        seed=int(rng.integers(1 << 62)), replica=r))
        fields.append(_polycrystal(e, e, e, c["Q"], 419, seed * 1000 + r))
    b = G.HMCBatch(shapes, c["Q"], per, c11=C11, c12=C12, c44=C44, kT=0.7, mpm_steps_per_mcs=c["mpm"],
                   precision=G.HMC_FP64 if c["precision"] == "fp64" else G.HMC_FP32)
    spins = torch.cat([f.reshape(-1) for f in fields])
    torch.cuda.synchronize()
    G.hmc_set_orientations_dev(b.h, _euler(c["Q"], seed), spins.data_ptr())
    return dict(case=c, h=b, fields=fields, outs=[torch.empty_like(f) for f in fields])


def _run_batch(s):
    b = s["h"]
    for r, f in enumerate(s["fields"]):
        b.select(r)
        G.hmc_set_spins_dev(b.h, f.data_ptr())
    accepted = b.mc_sweeps(s["case"]["mcs"])
    strains = []
    for r, o in enumerate(s["outs"]):
        strains.append(b.strain(r))
        G.hmc_get_spins_dev(b.h, o.data_ptr())
    strains = np.stack(strains)
    return dict(spins=s["outs"], accepted=accepted,
                strain=strains if s["case"]["precision"] == "fp64" else strains.astype(np.float32))


STRAIN6 = (-7.2e-4, -6.3e-4, 2e-3, 2e-4, -4e-4, 1e-4)


def _nodal(c, seed):
    """A nodal displacement and velocity field of the size that the solves meet, smooth over a few nodes."""
    g = torch.Generator(device=DEV).manual_seed(int(seed) + 7)
    f = torch.randn(2, c["nz"] // 2, c["ny"] // 2, c["nx"] // 2, 3, generator=g, device=DEV, dtype=torch.float64)
    for a in (1, 2, 3):
        f = f + 0.5 * (f.roll(1, a) + f.roll(-1, a))
    return f[0].reshape(-1, 3) * 1e-4, f[1].reshape(-1, 3) * 1e-6


def _prepare_solve(c, seed):
    spins = _polycrystal(c["nx"], c["ny"], c["nz"], c["Q"], c["grain"], seed)
    u, v = _nodal(c, seed)
    h = G.HMC((c["nz"], c["ny"], c["nx"]), c["Q"], c11=C11, c12=C12, c44=C44, bc=G.HMC_BC_STRAIN6, strain6=STRAIN6,
              precision=G.HMC_FP64 if c["precision"] == "fp64" else G.HMC_FP32)
    torch.cuda.synchronize()
    G.hmc_set_orientations_dev(h.h, _euler(c["Q"], seed), spins.data_ptr())
    return dict(case=c, h=h, u=u.cpu().numpy(), v=v.cpu().numpy())


def _run_solve(s):
    h = s["h"]
    h.set_nodal(s["u"], s["v"])
    energy = np.array([h.mpm_steps(s["case"]["steps"], want_energy=True)])
    u, v = h.nodal()
    t = np.float64 if s["case"]["precision"] == "fp64" else np.float32
    return dict(energy=energy.astype(t, copy=False), u=u.astype(t, copy=False), v=v.astype(t, copy=False))


def _prepare_stress(c, seed):
    spins = _polycrystal(c["nx"], c["ny"], c["nz"], c["Q"], c["grain"], seed)
    n = spins.numel()
    u = _nodal(c, seed)[0].float().contiguous()
    ctab = torch.from_numpy(_rotated(_euler(c["Q"], seed), (C11, C12, C44))).float().to(DEV).contiguous()
    f32, f64 = dict(device=DEV, dtype=torch.float32), dict(device=DEV, dtype=torch.float64)
    return dict(case=c, spins=spins, u=u, ctab=ctab, sigma=torch.empty(n, 6, **f32), mean=torch.empty(6, **f64),
                energy=torch.empty(1, **f64))


def _run_stress(s):
    c = s["case"]
    G.hmc_stress_noalloc(s["spins"].data_ptr(), s["u"].data_ptr(), s["ctab"].data_ptr(), STRAIN6, c["nx"], c["ny"],
                         c["nz"], s["sigma"].data_ptr(), s["mean"].data_ptr(), s["energy"].data_ptr(),
                         torch.cuda.current_stream().cuda_stream)
    return dict(sigma=s["sigma"], mean=s["mean"], energy=s["energy"])


def _prepare_adjoint(c, seed):
    spins = _polycrystal(c["nx"], c["ny"], c["nz"], c["Q"], c["grain"], seed).cpu().numpy().view(np.uint16)
    n = spins.size
    g = torch.Generator().manual_seed(int(seed) + 9)
    return dict(case=c, spins=spins, euler=_euler(c["Q"], seed),
                theta=torch.tensor((C11, C12, C44) + STRAIN6, dtype=torch.float64, requires_grad=True),
                weight=torch.rand(n, generator=g, dtype=torch.float64) / n)


def _run_adjoint(s):
    c = s["case"]
    W, w = HMCElastic.apply(s["theta"], s["spins"], s["euler"], c["steps"], c["checkpoint"],
                            G.HMC_FP64 if c["precision"] == "fp64" else G.HMC_FP32)
    (grad,) = torch.autograd.grad(W / w.numel() + (s["weight"] * w).sum(), s["theta"])
    t = torch.float64 if c["precision"] == "fp64" else torch.float32
    return dict(W=W.to(t), w=w.to(t), grad=grad.to(t))


def prepare(case, seed):
    return dict(mc=_prepare_mc, batch=_prepare_batch, solve=_prepare_solve, stress=_prepare_stress,
                adjoint=_prepare_adjoint)[case["kind"]](dict(case), int(seed))


def run(state):
    return dict(mc=_run_mc, batch=_run_batch, solve=_run_solve, stress=_run_stress,
                adjoint=_run_adjoint)[state["case"]["kind"]](state)


# ---- least work ---------------------------------------------------------------

POINT_STEP = 132.0   # flops of one point in one explicit step: gradients, strain, Hooke's law, forces, update


def work(case):
    c = case
    if c["kind"] == "batch":
        pool = [int(x) for x in c["edges"].split(",")]
        n = sum(pool[r % len(pool)] ** 3 for r in range(c["replicas"]))
    else:
        n = c["nx"] * c["ny"] * c["nz"]
    t = 8 if c.get("precision") == "fp64" else 4
    if c["kind"] in ("mc", "batch"):
        # spins in and out; displacement and velocity (six values a node, a node for eight sites) read
        # and written once where there are MPM steps; a random block a site and step
        state = 2 * 6 * t / 8 if c["mpm"] else 0
        return dict(bytes=n * (4 + state), flops=n * c["mcs"] * (POINT_STEP * c["mpm"] + 60.0))
    if c["kind"] == "solve":
        return dict(bytes=n * (2 + 2 * 6 * t / 8), flops=n * POINT_STEP * c["steps"])
    if c["kind"] == "stress":
        return dict(bytes=n * (2 + 1.5 + 24) + 144.0 * c["Q"], flops=n * 90.0)
    # forward steps, their reverse steps, and the parameter terms of each reverse step
    return dict(bytes=n * (2 + 2 * t), flops=n * c["steps"] * (2 * POINT_STEP + 100.0))


# ---- the same in 64 bits ------------------------------------------------------

def _rotated(euler, c):
    """(Q, 6, 6) Voigt stiffness of a cubic crystal (c11, c12, c44) in the sample frame."""
    out = np.zeros((len(euler), 6, 6))
    C = np.zeros((3, 3, 3, 3))
    for i in range(3):
        C[i, i, i, i] = c[0]
        for j in range(3):
            if i != j:
                C[i, i, j, j] = c[1]
                C[i, j, i, j] = C[i, j, j, i] = c[2]
    e = np.asarray(euler, dtype=np.float64)

    def rz(a):
        m = np.zeros((len(a), 3, 3))
        m[:, 0, 0] = m[:, 1, 1] = np.cos(a)
        m[:, 1, 0], m[:, 0, 1], m[:, 2, 2] = np.sin(a), -np.sin(a), 1.0
        return m

    ry = np.zeros((len(e), 3, 3))
    ry[:, 0, 0] = ry[:, 2, 2] = np.cos(e[:, 1])
    ry[:, 0, 2], ry[:, 2, 0], ry[:, 1, 1] = np.sin(e[:, 1]), -np.sin(e[:, 1]), 1.0
    A = rz(e[:, 0]) @ ry @ rz(e[:, 2])
    R = C[None]
    for a, b in (("qim,qmnop->qinop", "m"), ("qjn,qinop->qijop", "n"), ("qko,qijop->qijkp", "o"),
                 ("qlp,qijkp->qijkl", "p")):
        R = np.einsum(a, A, np.broadcast_to(R, (len(e), 3, 3, 3, 3)))
    for I in range(6):
        for J in range(6):
            out[:, I, J] = R[:, VI[I], VJ[I], VI[J], VJ[J]]
    return out


class _Elastic:
    """Cells of eight points (at 1/4 and 3/4 of each edge of a trilinear element of edge 2) on a periodic grid, in 64 bits."""

    def __init__(self, c, spins, tables):
        self.n = (c["nz"] // 2, c["ny"] // 2, c["nx"] // 2)
        nz, ny, nx = self.n
        s = spins.view(nz, 2, ny, 2, nx, 2).permute(0, 2, 4, 1, 3, 5).reshape(-1, 8).long()   # cell, point 4c+2b+a
        self.C = [t[s] for t in tables]              # (cells, 8, 6, 6) for each table
        grad = np.zeros((8, 8, 3))                   # corner, point, direction
        for corner in range(8):
            I = [corner & 1, corner >> 1 & 1, corner >> 2]
            for p in range(8):
                x = [(0.25, 0.75)[p >> a & 1] for a in range(3)]
                N = [x[a] if I[a] else 1 - x[a] for a in range(3)]
                for k in range(3):
                    grad[corner, p, k] = (0.5 if I[k] else -0.5) * N[(k + 1) % 3] * N[(k + 2) % 3]
        G6 = np.zeros((24, 48))                      # (corner, component) -> (point, Voigt strain)
        for corner in range(8):
            for d in range(3):
                for p in range(8):
                    for m in range(6):
                        i, j = VI[m], VJ[m]
                        if d == i:
                            G6[3 * corner + d, 6 * p + m] += grad[corner, p, j]
                        if d == j and i != j:
                            G6[3 * corner + d, 6 * p + m] += grad[corner, p, i]
        self.B = torch.from_numpy(G6).to(DEV)

    def strain(self, u, ebar):
        u = u.view(*self.n, 3)
        corners = [u.roll((-(c >> 2), -(c >> 1 & 1), -(c & 1)), (0, 1, 2)) for c in range(8)]
        return (torch.stack(corners, 3).reshape(-1, 24) @ self.B).view(-1, 8, 6) + ebar

    def stress(self, eps, theta):
        s = 0
        for t, C in zip(theta, self.C):
            s = s + t * (C * eps[:, :, None, :]).sum(-1)
        return s

    def force(self, sig):
        f = -(sig.reshape(-1, 48) @ self.B.T).view(*self.n, 8, 3)
        return sum(f[..., c, :].roll((c >> 2, c >> 1 & 1, c & 1), (0, 1, 2)) for c in range(8)).reshape(-1, 3)

    def step(self, u, v, theta, ebar):
        dt = 1.0 / math.sqrt(max(C11 + 2 * C12, C11 - C12, 2 * C44))   # half an element edge over the fastest wave
        v = 0.95 * v + dt / 8 * self.force(self.stress(self.strain(u, ebar), theta))
        return u + dt * v, v


def exact(case, seed):
    c = dict(case)
    if c["kind"] in ("mc", "batch"):
        return None      # whole numbers, and a mean strain that hangs on them
    spins = _polycrystal(c["nx"], c["ny"], c["nz"], c["Q"], c["grain"], seed)
    euler = _euler(c["Q"], seed)
    full = torch.from_numpy(_rotated(euler, (C11, C12, C44))).to(DEV)
    if c["kind"] == "stress":
        el = _Elastic(c, spins, [full.float().double()])
        u = _nodal(c, seed)[0].float().double()
        ebar = torch.tensor(STRAIN6, dtype=torch.float64, device=DEV).float().double()
        eps = el.strain(u, ebar)
        sig = el.stress(eps, [1.0])
        nz, ny, nx = el.n
        field = sig.view(nz, ny, nx, 2, 2, 2, 6).permute(0, 3, 1, 4, 2, 5, 6).reshape(-1, 6)
        return dict(sigma=field, mean=field.mean(0), energy=0.5 * (sig * eps).sum().reshape(1))
    ebar = torch.tensor(STRAIN6, dtype=torch.float64, device=DEV)
    if c["kind"] == "solve":
        el = _Elastic(c, spins, [full])
        u, v = _nodal(c, seed)
        for _ in range(c["steps"]):
            u, v = el.step(u, v, [1.0], ebar)
        eps = el.strain(u, ebar)
        return dict(energy=0.5 * (el.stress(eps, [1.0]) * eps).sum().reshape(1), u=u, v=v)
    basis = [torch.from_numpy(_rotated(euler, b)).to(DEV) for b in ((1, 0, 0), (0, 1, 0), (0, 0, 1))]
    el = _Elastic(c, spins, [full])
    rot = _Elastic(c, spins, basis) if c["nx"] * c["ny"] * c["nz"] <= 1 << 21 else None
    if rot is None:
        return None
    u = v = torch.zeros(math.prod(el.n), 3, dtype=torch.float64, device=DEV)
    past = []
    for _ in range(c["steps"]):
        past.append((u, v))
        u, v = el.step(u, v, [1.0], ebar)
    theta = torch.tensor((C11, C12, C44), dtype=torch.float64, device=DEV)
    g = torch.Generator().manual_seed(int(seed) + 9)
    n = spins.numel()
    weight = (torch.rand(n, generator=g, dtype=torch.float64) / n).to(DEV)

    def energy(u, theta, ebar):
        eps = rot.strain(u, ebar)
        w = 0.5 * (rot.stress(eps, theta) * eps).sum(-1)
        nz, ny, nx = el.n
        return w.view(nz, ny, nx, 2, 2, 2).permute(0, 3, 1, 4, 2, 5).reshape(-1)

    def back(out, ins):
        return torch.autograd.grad(out, ins)

    with torch.enable_grad():
        leaves = [x.detach().requires_grad_() for x in (u, theta, ebar)]
        w = energy(*leaves)
        gu, gt, ge = back(w.sum() / n + (weight * w).sum(), leaves)
        gv = torch.zeros_like(gu)
        for u, v in reversed(past):
            leaves = [x.detach().requires_grad_() for x in (u, v, theta, ebar)]
            un, vn = rot.step(*leaves)
            a, b, t, e = back((un * gu).sum() + (vn * gv).sum(), leaves)
            gu, gv, gt, ge = a, b, gt + t, ge + e
    w = w.detach()
    return dict(W=w.sum(), w=w, grad=torch.cat([gt, ge]))
