"""The default number of sweeps follows from the path that runs: 3 + 3 in 3D
where the V-cycles join a Krylov space, 6 + 6 on the paths without it (launch
modes 1 and 2, tile-streamed levels), 2 + 2 in 2D everywhere."""
import numpy as np
import pytest
import torch

from paper_1809_03745_gb300 import workloads as W

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1809_03745_gb300 import ebpoisson as E


@pytest.mark.parametrize("dim,path,nu", [(3, 0, 3), (3, 1, 6), (3, 2, 6), (3, "streamed", 6), (2, 0, 2), (2, 2, 2)])
def test_default_equals_the_stated_sweeps(dim, path, nu, monkeypatch):
    d = W.rod_plane_2d(64) if dim == 2 else W.pin_plane_3d(32, radius=0.13, disk_t=3.3 / 32)
    if path == "streamed":
        monkeypatch.setenv("EBP_SWEEP_MIN_CELLS", "1")
    g = E.Geometry(d)
    S = np.zeros((2, g.ncell))
    S[0] = np.random.default_rng(2).uniform(0, 50, g.ncell)
    out = []
    for kw in ({}, dict(nu1=nu, nu2=nu)):
        P = E.Poisson(g, tol=1e-10, max_cycles=400, launch_mode=0 if path == "streamed" else path, **kw)
        phi, info = P.solve(torch.from_numpy(S))
        assert info["status"] == 0 and (info["sweep_levels"] > 0) == (path == "streamed"), info
        out.append((phi, info["vcycles"]))
    assert out[0][1] == out[1][1]
    assert torch.equal(out[0][0], out[1][0])
