"""The colour-split persistent solve against the oracle where its parts change:
x rows that do not fill groups of four cells of a colour, coarse levels of odd
size (algebraic levels, one with a single row of cells), levels that lie in
one CTA or in the grid, V-cycles without pre- or post-smoothing, and FP64
residuals after one or several accelerated V-cycles.  Solves reach 1e-12 of
max|b|; the potential then agrees with the direct solution to 1e-9 like every
other parity case."""
import numpy as np
import pytest
import torch

import oracle
from paper_1809_03745_gb300 import workloads as W

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1809_03745_gb300 import ebpoisson as E


def _rod(nx, ny, dielectric):
    d = W.rod_plane_2d(nx, dielectric=dielectric, tip_y=0.5 * ny / nx, half_width=max(0.08, 3 / nx),
                       slab_y=0.2 * ny / nx + 0.3 / nx, rough_amp=0.0)
    d["n"] = (nx, ny, 1)
    return d


def _pin(nx, ny, nz, dielectric):
    d = W.pin_plane_3d(nx, tip_z=0.5 * nz / nx, radius=0.13, disk=dielectric, disk_t=3.3 / nx)
    d["n"] = (nx, ny, nz)
    return d


def _gap(n):
    return W._desc(len(n), n, (0.0,) * len(n), 1.0 / n[0], [], [], -1, -1, (1.0, 1.0),
                   [0, 0, 1, 1, 0, 0] if len(n) == 2 else [0, 0, 0, 0, 1, 1], 0.0, [0.0, 0.0, 0.0, 1.0, 0.0, 1.0])


CASES = {
    "rod_64x56": _rod(64, 56, True), "rod_104x72": _rod(104, 72, False), "rod_72x88": _rod(72, 88, True),
    "rod_200x136": _rod(200, 136, True), "rod_296x232": _rod(296, 232, False), "rod_512x488": _rod(512, 488, True),
    "pin_24x24x32": _pin(24, 24, 32, False), "pin_32x40x24": _pin(32, 40, 24, True), "pin_40x40x40": _pin(40, 40, 40, True),
    "gap_8x8": _gap((8, 8)), "gap_24x8": _gap((24, 8)), "gap_8x136": _gap((8, 136)), "gap_8x8x8": _gap((8, 8, 8)),
    "gap_24x8x40": _gap((24, 8, 40)),
}


def _fields(d, seed=3):
    x, y, z = W.cell_centres(d)
    rng = np.random.default_rng(seed)
    up = (y if d["dim"] == 2 else z) - 0.4 * d["n"][d["dim"] - 1] * d["h"]
    S = np.zeros((2, x.size))
    S[0] = 80.0 * np.exp(-((x - 0.45) ** 2 + up ** 2) / (2 * 0.05 ** 2)) + rng.uniform(-1, 1, x.size)
    S[1] = rng.uniform(-1, 1, x.size)
    return S, rng.uniform(-1, 1, x.size)


_cache = {}


def _oracle(name):
    if name not in _cache:
        S, sig = _fields(CASES[name])
        _cache[name] = (S, sig, oracle.solve(CASES[name], s=S, sigma=sig)[1])
    return _cache[name]


def _check(name, **opts):
    S, sig, want = _oracle(name)
    P = E.Poisson(E.Geometry(CASES[name]), tol=1e-12, max_cycles=400, **opts)
    phi, info = P.solve(torch.from_numpy(S), torch.from_numpy(sig))
    assert info["status"] == 0, info
    got = phi.cpu().numpy()
    assert np.abs(got - want).max() <= 1e-9 * np.abs(want).max(), info
    again, _ = P.solve(torch.from_numpy(S), torch.from_numpy(sig))
    assert torch.equal(phi, again)


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("name", list(CASES))
def test_solution_on_ragged_and_tiny_grids(name, precision):
    _check(name, precision=precision)


@pytest.mark.parametrize("opts", [dict(nu1=0), dict(nu2=0, nu1=4), dict(nu1=1, nu2=1), dict(inner_cycles=1),
                                  dict(inner_cycles=4), dict(bottom_sweeps=1)],
                         ids=lambda o: "_".join(f"{k}{v}" for k, v in o.items()))
@pytest.mark.parametrize("name", ["rod_200x136", "pin_40x40x40", "gap_24x8x40"])
def test_solution_with_other_cycles(name, opts):
    _check(name, **opts)
