"""The four-cell field pass and the FP32-first tags where they can go wrong:
caller pointers that are only 8-byte aligned (field and residuals), cell sizes
that are not powers of two (the corrected reciprocal against true division),
and tags at exact ties, at magnitudes outside FP32's range, on zero and on
infinite fields, against plain FP64 in numpy."""
import numpy as np
import pytest
import torch

from paper_1809_03745_gb300 import workloads as W

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1809_03745_gb300 import ebpoisson as E


def _problem(dim):
    if dim == 2:
        return W.rod_plane_2d(56, dielectric=True, rough_amp=0.0, slab_y=0.2 + 0.3 / 56)
    d = W.pin_plane_3d(24, radius=0.13, disk_t=3.3 / 24)
    d["n"] = (24, 24, 16)
    return d


def _shifted(t):
    """A copy of t whose data start 8 bytes off a 16-byte boundary."""
    buf = torch.empty(t.numel() + 1, dtype=t.dtype, device=t.device)
    out = buf[1:].view(t.shape)
    out.copy_(t)
    assert out.data_ptr() % 16 == 8
    return out


@pytest.mark.parametrize("dim", [2, 3])
def test_unaligned_pointers_give_the_same_bits(dim):
    d = _problem(dim)
    g = E.Geometry(d)
    P = E.Poisson(g, precision="fp64")
    n, neb = g.ncell, g.info["n_eb"]
    gen = torch.Generator(device="cuda").manual_seed(7)
    phi, rhs = (torch.randn(2, n, dtype=torch.float64, device="cuda", generator=gen) for _ in range(2))
    sig = torch.randn(n, dtype=torch.float64, device="cuda", generator=gen)
    got = []
    for f in (lambda t: t, _shifted):
        ph, r0, s0 = f(phi), f(rhs), f(sig)
        Ef = f(torch.zeros(dim, 2, n, dtype=torch.float64, device="cuda"))
        En = torch.zeros(neb, 2, dtype=torch.float64, device="cuda")
        E.eb_field_eval(P._h, ph, s0, Ef, En)
        r1, r2 = (f(torch.ones(2, n, dtype=torch.float64, device="cuda")) for _ in range(2))
        E.eb_poisson_residual(P._h, r0, s0, ph, r1)
        E.eb_poisson_residual_noalloc(g._h, r0, s0, ph, r2)
        got.append((Ef.clone(), En, r1.clone(), r2.clone()))
    for a, b in zip(*got):
        assert torch.equal(a, b)


@pytest.mark.parametrize("dim", [2, 3])
def test_regular_cells_carry_the_true_quotients(dim):
    d = _problem(dim)
    g = E.Geometry(d)
    P = E.Poisson(g, precision="fp64")
    n = [d["n"][k] for k in range(dim)]
    rng = np.random.default_rng(5)
    phi = rng.normal(size=(2, g.ncell)) * 10.0 ** rng.uniform(-12, 12, size=(2, g.ncell))
    Ef, _ = P.field(torch.from_numpy(phi))
    flags = g.export()["flags"].cpu().numpy().reshape(n[::-1])
    h = d["h"]
    for p in range(2):
        ph = phi[p].reshape(n[::-1])
        reg = (flags & 7) == (1 << p)
        for a in range(dim):
            ax = dim - 1 - a
            want = np.zeros_like(ph)
            c = np.moveaxis(ph, ax, 0)
            w = np.moveaxis(want, ax, 0)
            w[1:-1] = -(c[2:] - c[:-2]) / (2.0 * h)
            w[0] = -(c[1] - c[0]) / h
            w[-1] = -(c[-1] - c[-2]) / h
            got = Ef[a, p].cpu().numpy().reshape(n[::-1])
            assert np.array_equal(got[reg], want[reg])
    none = (flags & 3) == 0
    assert none.any() and not Ef.reshape(dim * 2, -1).cpu().numpy()[:, none.reshape(-1)].any()


def _tags(mag2, live, eps):
    """Tags and max |E| of a squared magnitude, in the order of the definition."""
    mag = np.sqrt(mag2) * live
    emax = mag.max()
    with np.errstate(all="ignore"):
        T = mag / emax if emax > 0 else np.zeros_like(mag)
        s2 = np.zeros_like(T)
        for ax in range(T.ndim - 1, -1, -1):  # x first
            t, lv = np.moveaxis(T, ax, 0), np.moveaxis(live, ax, 0)
            dd = np.zeros_like(t)
            hp, hm = np.zeros_like(lv), np.zeros_like(lv)
            hp[:-1], hm[1:] = lv[1:], lv[:-1]
            up, dn = np.zeros_like(t), np.zeros_like(t)
            up[:-1], dn[1:] = t[1:], t[:-1]
            dd = np.where(hp & hm, (up - dn) * 0.5, np.where(hp, up - t, np.where(hm, t - dn, 0.0)))
            s2 = s2 + np.moveaxis(dd * dd, 0, ax)
        g = np.sqrt(s2)
        ratio = np.where(T > 0, g / T, np.where(g > 0, np.inf, 0.0))
        tags = ((ratio > eps[0]) | (T > eps[1])) * 1 + ((ratio < eps[2]) & (T < eps[3])) * 2
    return (tags * live).astype(np.uint8), emax


@pytest.mark.parametrize("kind", ["ties", "tiny", "huge", "mixed", "zero", "wide"])
@pytest.mark.parametrize("dim", [2, 3])
def test_tags_equal_plain_fp64(dim, kind):
    d = _problem(dim)
    d = dict(d, prims=[], nodes=[], root_E=-1, root_D=-1, electrodes=[])  # every cell a gas cell
    g = E.Geometry(d)
    n = [d["n"][k] for k in range(dim)]
    rng = np.random.default_rng(11)
    i = np.indices(n[::-1])[-1].astype(float)
    base = 1.0 + i / 64.0  # ratio and T sit on representable values: ties with the thresholds below
    if kind in ("tiny", "huge"):
        base = base * (1e-30 if kind == "tiny" else 1e30) * rng.uniform(0.5, 1.5, base.shape)
    if kind == "mixed":
        base = 10.0 ** rng.uniform(-25, 0, base.shape)
    if kind == "zero":
        base = base * (rng.uniform(size=base.shape) < 0.3)
    if kind == "wide":
        base = rng.uniform(0.0, 1.0, base.shape) ** 2
    Ef = np.zeros((dim, 2, base.size))
    Ef[0, 0] = base.reshape(-1)
    eps = (0.1, 0.8, 0.1, 0.2)
    if kind == "ties":
        T = base / base.max()
        row = T.reshape(-1, n[0])[0]
        eps = (float((row[9] - row[7]) * 0.5 / row[8]), float(row[20]), float((row[9] - row[7]) * 0.5 / row[8]), float(row[20]))
    tags, _, _, marked, emax = E.tag_cells(g, torch.from_numpy(Ef).cuda(), eps=eps)
    want, want_max = _tags((base * base), np.ones(base.shape, bool), eps)
    assert np.array_equal(tags.cpu().numpy(), want.reshape(-1))
    assert marked == int((want & 1).sum()) and emax == want_max
