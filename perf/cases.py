"""The work that a user of the solver has it do, as measurable cases.

Each case is one call (or the few calls that belong together) of the public
Python API on inputs that are already where a plasma code has them: on the GPU,
next to the geometry and solver handles that such a code keeps from step to
step.  The server case starts from host arrays, as a serving client does.

Solves run to the tight tolerances (1e-12 and 1e-13 of max|b|) at which the
solver's own parity runs compare potentials: there the potential is settled to
more than nine digits on every grid, the slowly converging ones too, so it
does not depend on the path that the iteration took.

The geometries are the rod-plane (2D) and pin-plane (3D) electrodes of
workloads.py, with or without a dielectric, the plane gap without bodies, and
the refined box around the tip.  Grids need not be square or powers of two:
any extent that is a multiple of 8 is accepted and used.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1809_03745_gb300 import ebpoisson as E
from paper_1809_03745_gb300 import photoionization as PH
from paper_1809_03745_gb300 import workloads as W

TOL = 1e-13  # potentials: max|b| is that of the wall data, far above the rounding of A phi
TOL_SHIFT = 1e-12  # Helmholtz solves: max|b| is that of the source, nearer to it
MAX_CYCLES = 800


def listed():
    return [
        # the smallest solve in use (the vacuum rod-plane test problem): all latency
        dict(name="rod2d_128", kind="solve", dim=2, nx=128, ny=128, nz=1, dielectric=False, precision="mixed"),
        # the multi-material 2D workload: rough dielectric, surface charge, one solve of a time step
        dict(name="rod2d_1024", kind="solve", dim=2, nx=1024, ny=1024, nz=1, dielectric=True, precision="mixed"),
        # a 2D grid whose extents halve only three times: coarsening stops early
        dict(name="rod2d_632x488", kind="solve", dim=2, nx=632, ny=488, nz=1, dielectric=True, precision="mixed"),
        # FP64 V-cycles, the solver's other precision option
        dict(name="rod2d_512_fp64", kind="solve", dim=2, nx=512, ny=512, nz=1, dielectric=True, precision="fp64"),
        # the 3D pin-plane with a dielectric disk on a single grid
        dict(name="pin3d_256", kind="solve", dim=3, nx=256, ny=256, nz=256, dielectric=True, precision="mixed"),
        # the largest single grid of the serving mix
        dict(name="pin3d_384", kind="solve", dim=3, nx=384, ny=384, nz=384, dielectric=True, precision="mixed"),
        # the 3D pin-plane with a ratio-2 box around the tip (the headline workload)
        dict(name="composite3d_256", kind="composite", n=256),
        # many small independent solves in one call (parameter scans)
        dict(name="batch_20", kind="batch", count=20, mix=4, n2_max=512, n3_max=112),
        # one implicit diffusion step: two Helmholtz solves
        dict(name="tga2d_1024", kind="tga", dim=2, n=1024, r=10.0),
        # one photoionisation update in a plane gap: three Helmholtz solves with Robin walls
        dict(name="photo3d_gap", kind="photo", nx=152, ny=136, nz=200),
        # field and refinement tags of a 3D grid, as between two regrids
        dict(name="field_tags_256", kind="field", nx=256, ny=256, nz=256),
        # a burst of requests through the server: geometry, hierarchy and solve of each
        dict(name="serve_12", kind="serve", count=12, mix=5, n2_max=320, n3_max=64),
    ]


def _n8(rng, lo, hi):
    """A multiple of 8, spread over the logarithm of [lo, hi]."""
    return max(lo, min(hi, 8 * int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / 8))))


def _near(rng, n, top, least=0.75):
    return max(40, min(top, 8 * int(round(n * rng.uniform(least, 1.25) / 8))))


def draw(rng):
    kind = rng.choice(["solve2", "solve2", "solve3", "solve3", "composite", "batch", "tga", "photo", "field", "serve"])
    if kind == "solve2":
        nx = _n8(rng, 64, 1024)
        return dict(kind="solve", dim=2, nx=nx, ny=_near(rng, nx, 1024), nz=1, dielectric=rng.random() < 0.6,
                    precision="fp64" if rng.random() < 0.25 else "mixed")
    if kind == "solve3":
        nx = _n8(rng, 48, 352)
        n = (nx, _near(rng, nx, 384, 0.95), _near(rng, nx, 384))
        if nx > 200:  # large grids are chosen to halve a few times
            n = tuple(16 * (v // 16) for v in n)
            n = (n[0], max(n[0], n[1]), n[2])
        return dict(kind="solve", dim=3, nx=n[0], ny=n[1], nz=n[2],
                    dielectric=rng.random() < 0.6, precision="mixed")
    if kind == "composite":
        return dict(kind="composite", n=16 * rng.randint(4, 15))
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(6, 24), mix=rng.randrange(1 << 20), n2_max=8 * rng.randint(16, 64),
                    n3_max=8 * rng.randint(6, 14))
    if kind == "tga":
        dim = rng.choice([2, 3])
        return dict(kind="tga", dim=dim, n=16 * int(round(_n8(rng, 96, 1008) / 16)) if dim == 2 else 16 * rng.randint(4, 12),
                    r=10.0 ** rng.uniform(-1.0, 2.5))
    if kind == "photo":
        nx = _n8(rng, 48, 232)
        return dict(kind="photo", nx=nx, ny=_near(rng, nx, 256), nz=_near(rng, nx, 256))
    if kind == "field":
        nx = _n8(rng, 48, 240)
        return dict(kind="field", nx=nx, ny=_near(rng, nx, 256, 0.95), nz=_near(rng, nx, 256))
    return dict(kind="serve", count=rng.randint(4, 12), mix=rng.randrange(1 << 20), n2_max=8 * rng.randint(12, 40),
                n3_max=8 * rng.randint(5, 8))


# ------------------------------------------------------------------ problems

def _problem(case):
    """The description of a single-grid case: cells of 1/nx, the tip at half the
    gap.  (The disk's edge is at 0.8, so y reaches past 0.9 in 3D.)"""
    n = (case["nx"], case["ny"]) + ((case["nz"],) if case["dim"] == 3 else ())
    h = 1.0 / n[0]
    top = n[-1] * h
    if case["dim"] == 2:
        # the slab's roughness needs a few cells per period, and coarse grids that follow it down
        rough = 0.005 if n[0] >= 512 and n[0] % 64 == 0 and n[1] % 64 == 0 else 0.0
        slab = 0.2 if rough else 0.2 + 0.3 * h
        d = W.rod_plane_2d(n[0], dielectric=case["dielectric"], tip_y=0.5 * top, half_width=max(0.05, 3 * h),
                           slab_y=slab, rough_amp=rough)
    else:
        d = W.pin_plane_3d(n[0], tip_z=0.5 * top, radius=max(0.02, 3 * h), disk=case["dielectric"],
                           disk_t=max(0.05, 3 * h) + 0.3 * h)
    d["n"] = tuple(n) + (1,) * (3 - len(n))
    return d


def _axes(d, dev):
    """Cell-centre coordinates that broadcast over the grid (z, y, x)."""
    ax = [d["lo"][k] + (torch.arange(d["n"][k], dtype=torch.float64, device=dev) + 0.5) * d["h"] for k in range(3)]
    if d["dim"] == 2:
        return ax[0][None, None, :], ax[1][None, :, None], torch.zeros(1, 1, 1, dtype=torch.float64, device=dev)
    return ax[0][None, None, :], ax[1][None, :, None], ax[2][:, None, None]


class _Seeded:
    """Numbers of one seed: scalars from numpy, fields from torch."""

    def __init__(self, seed, dev):
        self.np = np.random.Generator(np.random.PCG64(seed))
        self.dev = dev
        self.g = torch.Generator(device=dev)
        self.g.manual_seed(int(seed) + 977)

    def u(self, a, b):
        return float(self.np.uniform(a, b))

    def logu(self, a, b):
        return math.exp(self.u(math.log(a), math.log(b)))

    def field(self, n, a, b):
        return torch.rand(n, generator=self.g, dtype=torch.float64, device=self.dev) * (b - a) + a


def _charges(d, q, dev, tip=None):
    """Space charge of a discharge head below the tip and its trail on the
    axis, with a little noise, and a surface charge per cell (read on
    dielectric interfaces only)."""
    x, y, z = _axes(d, dev)
    up = y if d["dim"] == 2 else z
    side = (x - 0.5) ** 2 + ((y - 0.5) ** 2 if d["dim"] == 3 else 0.0)
    if tip is None:
        p = d["prims"][0][1]
        tip = p[d["dim"] - 1] - p[6]
    head, w, trail = tip - q.u(0.03, 0.1), q.u(0.02, 0.035), q.u(0.1, 0.5)
    s = q.logu(50.0, 800.0) * (torch.exp(-(side + (up - head) ** 2) / (2 * w * w))
                               + trail * torch.exp(-side / (2 * w * w)) * (up < tip) * (up > 0.5 * tip))
    n = W.ncells(d)
    S = torch.zeros(2, n, dtype=torch.float64, device=dev)
    S[0] = s.expand(d["n"][2], d["n"][1], d["n"][0]).reshape(-1) + q.field(n, -1e-3, 1e-3)
    return S, q.field(n, -1.0, 1.0)


def _instances(case):
    """The descriptions of a batch or a burst: 2D or 3D, sizes log-uniform, the
    electrode, gap, dielectric and voltage drawn, every feature at least
    three cells thick."""
    rng = np.random.Generator(np.random.PCG64(case["mix"]))
    out = []
    for k in range(case["count"]):
        dim = 3 if rng.uniform() < 0.5 else 2
        lo, hi = (32, case["n3_max"]) if dim == 3 else (64, case["n2_max"])
        n = max(lo, 8 * int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / 8)))
        h = 1.0 / n
        tip_r, gap = max(rng.uniform(0.01, 0.05), 3 * h), rng.uniform(0.4, 0.7)
        eps, V = rng.uniform(2.0, 8.0), rng.uniform(0.5, 2.0)
        thick = max(min(0.05 if dim == 3 else 0.1, gap - 10 * h), 3 * h) + 0.3 * h
        if dim == 3:
            d = W.pin_plane_3d(n, tip_z=gap, radius=tip_r, V=V, eps_d=eps, disk_t=thick)
        else:
            d = W.rod_plane_2d(n, dielectric=True, tip_y=gap, half_width=tip_r, V=V, eps_d=eps, slab_y=thick,
                               rough_amp=0.0)
        out.append(d)
    return out


PHOTO_L = 0.02  # edge of the photoionisation box in metres, along x


def _gap_group(case, group):
    """One photon group in a plane gap without bodies: every wall absorbs."""
    kl = W.photo_kappa(group) * PHOTO_L
    a1 = 1.5 * kl
    return dict(dim=3, n=(case["nx"], case["ny"], case["nz"]), lo=(0.0, 0.0, 0.0), h=1.0 / case["nx"], prims=[],
                nodes=[], root_E=-1, root_D=-1, electrodes=[], eps=(1.0, 1.0), bc=[W.ROBIN] * 6, phi_E=0.0,
                phi_wall=[0.0] * 6, robin=[(a1, 1.0)] * 6, lam=(3.0 * kl * kl, 0.0))


def _emission(case, seed, dev):
    """The three groups' sources 3 kappa L^2 eta of one emission region."""
    q = _Seeded(seed, dev)
    d = _gap_group(case, 0)
    x, y, z = _axes(d, dev)
    ly, lz = case["ny"] * d["h"], case["nz"] * d["h"]
    w = q.u(0.03, 0.06)
    eta = q.logu(0.3, 3.0) * torch.exp(-((x - q.u(0.4, 0.6)) ** 2 + (y - q.u(0.4, 0.6) * ly) ** 2
                                         + (z - q.u(0.3, 0.7) * lz) ** 2) / (2 * w * w))
    eta = eta.reshape(-1) + q.field(W.ncells(d), 0.0, 1e-4)
    out = []
    for k in range(3):
        S = torch.zeros(2, W.ncells(d), dtype=torch.float64, device=dev)
        S[0] = 3.0 * W.photo_kappa(k) * PHOTO_L ** 2 * eta
        out.append(S)
    return out


def _photo_weights():
    return [W.PHOTO_NU_EFF * W.PHOTO_P_O2 * W.PHOTO_GROUPS[k][1] for k in range(3)]


# ------------------------------------------------------------------ the cases

def _poisson(d, precision="mixed", tol=TOL):
    return E.Poisson(E.Geometry(d), precision=precision, tol=tol, max_cycles=MAX_CYCLES)


def prepare(case, seed):
    dev = torch.device("cuda")
    kind = case["kind"]
    q = _Seeded(seed, dev)
    if kind == "solve":
        d = _problem(case)
        S, sig = _charges(d, q, dev)
        return dict(kind=kind, P=_poisson(d, case["precision"]), S=S, sig=sig)
    if kind == "composite":
        n = case["n"]
        d = W.pin_plane_3d(n, radius=max(0.02, 3.0 / n), disk_t=max(0.05, 3.0 / n) + 0.3 / n)
        lo, hi = [3 * n // 8 // 4 * 4] * 3, [3 * n // 8 // 4 * 4 + n // 4] * 3
        C = E.Composite(d, lo, hi, tol=TOL, max_cycles=MAX_CYCLES)
        # the same head on both grids: the numbers are drawn once more from the same seed
        Sc, sc = _charges(d, q, dev)
        Sf, sf = _charges(W.refined_box_desc(d, lo, hi), _Seeded(seed, dev), dev)
        return dict(kind=kind, C=C, args=(Sc, Sf, sc, sf))
    if kind == "batch":
        ds = _instances(case)
        data = [_charges(d, q, dev) for d in ds]
        return dict(kind=kind, P=[_poisson(d) for d in ds], S=[v[0] for v in data], sig=[v[1] for v in data])
    if kind == "tga":
        n, dim = case["n"], case["dim"]
        d, _, _ = W.diffusion_inputs(dim, 8)  # the geometry of that workload at this size
        big = W.rod_plane_2d(n, dielectric=True, rough_amp=0.005 if n % 512 == 0 else 0.0,
                             slab_y=0.2 if n % 512 == 0 else 0.2 + 0.3 / n) if dim == 2 else \
            W.pin_plane_3d(n, radius=max(0.02, 3.0 / n), disk_t=max(0.05, 3.0 / n) + 0.3 / n)
        d.update(n=big["n"], h=big["h"], prims=big["prims"])
        T = E.TGA(d, case["r"] / float(n) ** 2, tol=TOL_SHIFT)
        kap = T.geom.export()["kappa"]
        phi = _charges(d, q, dev)[0] * (kap > 0)
        rho = _charges(d, q, dev)[0] * (kap > 0)
        return dict(kind=kind, T=T, phi=phi, rho=rho)
    if kind == "photo":
        solvers = []
        for k, S in enumerate(_emission(case, seed, dev)):
            P = _poisson(_gap_group(case, k), tol=TOL_SHIFT)
            solvers.append((P.geom, P, S, None))
        return dict(kind=kind, solvers=solvers, w=_photo_weights())
    if kind == "field":
        d = _problem(dict(case, dim=3, dielectric=True))
        P = _poisson(d)
        x, y, z = _axes(d, dev)
        top = d["n"][2] * d["h"]
        # a potential like the solved one: the gap's gradient, steep at the tip, and smooth waves of space charge
        r = torch.sqrt((x - 0.5) ** 2 + (y - 0.5) ** 2 + (z - 0.5 * top) ** 2 + 1e-4)
        phi = z / top + q.u(0.01, 0.03) / (r + 0.02)
        for _ in range(4):
            phi = phi + q.u(-0.02, 0.02) * torch.sin(q.u(2, 9) * x + q.u(2, 9) * y + q.u(2, 9) * z + q.u(0, 6))
        n = W.ncells(d)
        return dict(kind=kind, P=P, phi=phi.reshape(1, n).expand(2, n).contiguous(), sig=q.field(n, -1.0, 1.0))
    if kind == "serve":
        ds = _instances(case)
        reqs = []
        for d in ds:
            S, sig = _charges(d, q, dev)
            reqs.append((d, S.cpu().numpy(), sig.cpu().numpy()))
        return dict(kind=kind, server=E.Server(max_slots=64, tol=TOL, max_cycles=MAX_CYCLES), reqs=reqs)
    raise ValueError(kind)


def run(state):
    kind = state["kind"]
    if kind == "solve":
        return state["P"].solve(state["S"], state["sig"])[0]
    if kind == "composite":
        return list(state["C"].solve(*state["args"])[:2])
    if kind == "batch":
        return E.solve_batched(state["P"], state["S"], state["sig"])[0]
    if kind == "tga":
        return state["T"].step(state["phi"], state["rho"])[0]
    if kind == "photo":
        psi, sph, _ = PH.update(state["solvers"], state["w"])
        return dict(psi=psi, sph=sph)
    if kind == "field":
        P = state["P"]
        Ef, En = P.field(state["phi"], state["sig"])
        tags, lo, hi, marked, emax = E.tag_cells(P.geom, Ef)
        return dict(E=Ef, En=En, tags=tags, box=lo + hi, marked=marked, emax=emax)
    server = state["server"]
    tickets = [server.submit(*r) for r in state["reqs"]]
    return [server.wait(t)[0] for t in tickets]


# ------------------------------------------------------------------ yardsticks

def _cells(d):
    return float(W.ncells(d))


def _solve_work(n, dim, phases):
    """One solve: each phase's charge and (with a dielectric) the surface
    charge read, the potential written; and the arithmetic of a multigrid that
    gains a decimal digit per V-cycle of four sweeps, a residual and two
    transfers, 13 digits over the levels."""
    return dict(bytes=n * 8.0 * (phases + (phases - 1) + 2),
                flops=13 * 6 * (4 * dim + 3) * n / (1.0 - 0.5 ** dim))


def work(case):
    kind = case["kind"]
    if kind == "solve":
        n = float(case["nx"]) * case["ny"] * case["nz"]
        return _solve_work(n, case["dim"], 2 if case["dielectric"] else 1)
    if kind == "composite":
        return _solve_work(float(case["n"]) ** 3 + (case["n"] / 2.0) ** 3, 3, 2)
    if kind in ("batch", "serve"):
        parts = [_solve_work(_cells(d), d["dim"], 2) for d in _instances(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    if kind == "tga":
        # two stage solves, the state and the source read, the next state written
        n = float(case["n"]) ** case["dim"]
        return dict(bytes=n * 8.0 * 4, flops=2 * _solve_work(n, case["dim"], 1)["flops"])
    if kind == "photo":
        n = float(case["nx"]) * case["ny"] * case["nz"]
        w = _solve_work(n, 3, 1)
        return dict(bytes=3 * w["bytes"] + 8.0 * n, flops=3 * w["flops"])
    # field: the potential read, three components of both phases written, read again for the tags
    n = float(case["nx"]) * case["ny"] * case["nz"]
    return dict(bytes=n * (16.0 + 48.0 + 8.0 + 1.0), flops=n * 40.0)


def exact(case, seed):
    """The discrete solution by separation of variables where the operator is
    separable: the plane gap without bodies.  The other geometries' cut cells
    have no plain formula; None for those."""
    if case["kind"] != "photo":
        return None
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    psi = []
    for k, S in enumerate(_emission(case, seed, dev)):
        d = _gap_group(case, k)
        h, a1 = d["h"], d["robin"][0][0]
        w = a1 / (a1 + 8.0 / (3.0 * h))  # what the one-sided wall formula leaves of a wall value with a2 = 1
        lam, left, right = [], [], []
        for n in d["n"]:
            A = np.zeros((n, n))
            for i in range(n):
                if i > 0:
                    A[i, i - 1] -= 1.0
                    A[i, i] += 1.0
                if i < n - 1:
                    A[i, i + 1] -= 1.0
                    A[i, i] += 1.0
            A[0, 0] += 3.0 * w
            A[0, 1] -= w / 3.0
            A[n - 1, n - 1] += 3.0 * w
            A[n - 1, n - 2] -= w / 3.0
            sc = np.ones(n)  # diag(sc) A diag(1/sc) is symmetric: only the first and last rows are not
            sc[0] = sc[n - 1] = 1.0 / math.sqrt(1.0 + w / 3.0)
            ev, Q = np.linalg.eigh(sc[:, None] * A / sc[None, :])
            t = lambda v: torch.from_numpy(np.ascontiguousarray(v)).to(dev)  # noqa: E731
            lam.append(t(ev))
            left.append(t(Q.T * sc[None, :]))
            right.append(t(Q / sc[:, None]))
        nx, ny, nz = d["n"]
        u = S[0].reshape(nz, ny, nx)
        u = torch.einsum("ai,kji->kja", left[0], u)
        u = torch.einsum("aj,kji->kai", left[1], u)
        u = torch.einsum("ak,kji->aji", left[2], u)
        u = u / ((lam[0][None, None, :] + lam[1][None, :, None] + lam[2][:, None, None]) / (h * h) + d["lam"][0])
        u = torch.einsum("ia,kja->kji", right[0], u)
        u = torch.einsum("ja,kai->kji", right[1], u)
        u = torch.einsum("ka,aji->kji", right[2], u)
        p = torch.zeros(2, nx * ny * nz, dtype=torch.float64, device=dev)
        p[0] = u.reshape(-1)
        psi.append(p)
    return dict(psi=psi, sph=sum(wg * p[0] for wg, p in zip(_photo_weights(), psi)))
