"""The benchmark hook: the tile-streamed kernels (4, 5) are timed on every
handle whose finest grid is large enough for them, and on a smaller one that
was built to stream."""
import pytest
import torch

from paper_1809_03745_gb300 import workloads as W

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1809_03745_gb300 import ebpoisson as E


def _gap(n):
    return W._desc(3, n, (0.0, 0.0, 0.0), 1.0 / n[0], [], [], -1, -1, (1.0, 1.0), [0, 0, 0, 0, 1, 1], 0.0,
                   [0.0, 0.0, 0.0, 0.0, 0.0, 1.0])


@pytest.mark.parametrize("dielectric", [False, True])
def test_streamed_kernels_from_2_25_cells_on(dielectric):
    n = (512, 256, 256)
    d = W.pin_plane_3d(512, tip_z=0.3, radius=0.02, disk_t=0.1) if dielectric else _gap(n)
    d["n"] = n
    P = E.Poisson(E.Geometry(d), precision="mixed", tol=1e-8)
    S = torch.zeros(2, P.geom.ncell, dtype=torch.float64, device="cuda")
    S[0] = 1.0
    before, info = P.solve(S)
    for kernel, per in ((4, 13.0), (5, 10.0)):
        ms, by = P.profile(kernel, reps=2)
        assert ms > 0.0 and by == per * P.geom.ncell
    after, again = P.solve(S)  # the handle solves as before
    assert torch.equal(before, after) and again["vcycles"] == info["vcycles"] and info["status"] == 0


def test_streamed_kernels_refused_where_there_are_none(monkeypatch):
    small = E.Geometry(W.pin_plane_3d(32, radius=0.13))
    wide = E.Geometry(_gap((520, 256, 256)))  # x not a multiple of 16
    big = E.Geometry(_gap((512, 256, 256)))
    for g, kw in ((small, {}), (wide, {}), (big, dict(precision="fp64")), (big, dict(launch_mode=2))):
        P = E.Poisson(g, **kw)
        for kernel in (4, 5):
            with pytest.raises(E.EBError) as exc:
                P.profile(kernel, reps=1)
            assert exc.value.status == E.EB_ERR_UNSUPPORTED
    P = E.Poisson(big)
    monkeypatch.setenv("EBP_SWEEP", "0")
    with pytest.raises(E.EBError):
        P.profile(4, reps=1)
    monkeypatch.delenv("EBP_SWEEP")
    monkeypatch.setenv("EBP_SWEEP_MIN_CELLS", "1")
    assert E.Poisson(small).profile(4, reps=1)[0] > 0.0
