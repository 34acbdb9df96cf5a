"""The server's estimate of a request's memory, made before it is built, is an
upper bound for both precisions with a dielectric that fills most of the grid
(its vectors are stored for nearly every cell), in 2D and 3D, and admission by
it keeps to the budget."""
import numpy as np
import pytest
import torch

from paper_1809_03745_gb300 import workloads as W

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1809_03745_gb300 import ebpoisson as E


def _thick(dim, n, dielectric):
    if dim == 2:
        return W.rod_plane_2d(n, dielectric=dielectric, tip_y=0.9, slab_y=0.8 + 0.3 / n, rough_amp=0.0)
    return W.pin_plane_3d(n, tip_z=0.92, radius=max(0.02, 3 / n), disk=dielectric, disk_t=0.8 + 0.3 / n, disk_r=0.45)


@pytest.mark.parametrize("dielectric", [False, True])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("dim,n", [(2, 64), (2, 1024), (3, 32), (3, 120)])
def test_estimate_is_an_upper_bound(dim, n, precision, dielectric):
    d = _thick(dim, n, dielectric)
    S = np.zeros((2, W.ncells(d)))
    S[0] = 1.0
    srv = E.Server(max_slots=1, precision=precision, tol=1e-6, max_cycles=400)
    try:
        _, info = srv.wait(srv.submit(d, S, None), 300.0)
        st = srv.stats()
    finally:
        srv.close()
    assert info["status"] == 0, info
    assert st["estimate_misses"] == 0, st


def test_budget_holds_with_fp64_cycles_and_a_thick_dielectric():
    d = _thick(2, 512, True)
    S = np.zeros((2, W.ncells(d)))
    S[0] = 1.0
    srv = E.Server(max_slots=8, hbm_budget_bytes=2.5e8, precision="fp64", tol=1e-6, max_cycles=400)
    try:
        res = [srv.wait(t, 300.0) for t in [srv.submit(d, S, None) for _ in range(6)]]
        st = srv.stats()
    finally:
        srv.close()
    assert all(r[1]["status"] == 0 for r in res)
    assert st["estimate_misses"] == 0 and st["hbm_peak"] <= st["hbm_budget"], st
