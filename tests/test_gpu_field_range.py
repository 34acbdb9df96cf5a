"""The field at the ends of FP64's range: the regular cells carry the true
quotients where these overflow, are subnormal or are zeros of either sign, and
an infinite field is tagged as plain FP64 has it."""
import numpy as np
import pytest
import torch

from test_gpu_field_tags_edge import _problem, _tags

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1809_03745_gb300 import ebpoisson as E


def _bits(a):
    return np.ascontiguousarray(a).view(np.uint64)


@pytest.mark.parametrize("kind", ["overflow", "subnormal", "zeros", "infinite"])
@pytest.mark.parametrize("dim", [2, 3])
def test_regular_cells_carry_the_true_quotients(dim, kind):
    d = _problem(dim)
    d = dict(d, prims=[], nodes=[], root_E=-1, root_D=-1, electrodes=[])  # every cell a regular gas cell
    g = E.Geometry(d)
    P = E.Poisson(g, precision="fp64")
    n = [d["n"][k] for k in range(dim)]
    rng = np.random.default_rng(23)
    phi = np.zeros((2, g.ncell))
    u = rng.normal(size=g.ncell)
    if kind == "overflow":
        phi[0] = u * 10.0 ** rng.uniform(304, 307, g.ncell)
    elif kind == "subnormal":
        phi[0] = u * 10.0 ** rng.uniform(-323, -300, g.ncell)
    elif kind == "zeros":
        phi[0] = rng.integers(0, 2, g.ncell) * rng.choice([-1.0, 1.0], g.ncell) * np.round(u)
    else:
        phi[0] = np.where(rng.uniform(size=g.ncell) < 0.1, np.inf, u)
    Ef, _ = P.field(torch.from_numpy(phi))
    h, ph = d["h"], phi[0].reshape(n[::-1])
    with np.errstate(all="ignore"):
        for a in range(dim):
            c = np.moveaxis(ph, dim - 1 - a, 0)
            want = np.empty_like(c)
            want[1:-1] = -(c[2:] - c[:-2]) / (2.0 * h)
            want[0] = -(c[1] - c[0]) / h
            want[-1] = -(c[-1] - c[-2]) / h
            got = np.moveaxis(Ef[a, 0].cpu().numpy().reshape(n[::-1]), dim - 1 - a, 0)
            nan = np.isnan(want)
            assert np.array_equal(np.isnan(got), nan)
            assert np.array_equal(_bits(got[~nan]), _bits(want[~nan]))
            if kind == "overflow":
                assert np.isinf(want).any() and np.isfinite(want).any()


@pytest.mark.parametrize("dim", [2, 3])
def test_infinite_field_is_tagged_as_plain_fp64_has_it(dim):
    d = _problem(dim)
    d = dict(d, prims=[], nodes=[], root_E=-1, root_D=-1, electrodes=[])
    g = E.Geometry(d)
    n = [d["n"][k] for k in range(dim)]
    base = np.random.default_rng(29).uniform(0.1, 1.0, n[::-1])
    base.reshape(-1)[[3, g.ncell // 2]] = np.inf
    Ef = np.zeros((dim, 2, base.size))
    Ef[0, 0] = base.reshape(-1)
    eps = (0.1, 0.8, 0.1, 0.2)
    tags, _, _, marked, emax = E.tag_cells(g, torch.from_numpy(Ef).cuda(), eps=eps)
    want, want_max = _tags(base * base, np.ones(base.shape, bool), eps)
    assert np.array_equal(tags.cpu().numpy(), want.reshape(-1))
    assert marked == int((want & 1).sum()) and emax == want_max == np.inf
