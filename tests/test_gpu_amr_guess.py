"""A composite solve returns 0 in the entries without an unknown, whatever the
initial guess held there (a buffer used before, or never written), and the
same potential elsewhere."""
import numpy as np
import pytest
import torch

from paper_1809_03745_gb300 import workloads as W

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1809_03745_gb300 import ebpoisson as E


@pytest.mark.parametrize("dielectric", [False, True])
@pytest.mark.parametrize("boxes", [1, 2])
@pytest.mark.parametrize("warm", [False, True])
@pytest.mark.parametrize("junk", [7.0, float("nan")])
def test_entries_without_an_unknown_come_out_zero(dielectric, boxes, warm, junk):
    d = W.rod_plane_2d(64, dielectric=dielectric, rough_amp=0.0, slab_y=0.1 + 0.3 / 64)
    H = E.Hierarchy(d, [([24, 24], [40, 40]), ([8, 8], [24, 24])][:boxes], tol=1e-12, max_cycles=100)
    rng = np.random.default_rng(31)
    rhs, absent = [], []
    for l in range(H.L):
        S = np.zeros((2, H.levels[l]["n_cells"]))
        S[0] = rng.uniform(0, 100, S.shape[1])
        rhs.append(torch.from_numpy(S).cuda())
        f = E.Geometry(H.level_desc(l)).export()["flags"]
        absent.append(torch.stack([(f & 1) == 0, (f & 2) == 0]))
        assert absent[l].any()
    want, info = H.solve(rhs)
    assert info["status"] == 0, info
    guess = [torch.where(a, junk, t if warm else 0.0 * t) for t, a in zip(want, absent)]
    got, info = H.solve(rhs, phi=guess)
    assert info["status"] == 0, info
    for g, w, a in zip(got, want, absent):
        assert not w[a].any()
        assert not torch.isnan(g).any() and not g[a].any()
        assert (g - w).abs().max() <= 1e-9 * w.abs().max()  # as every parity case at 1e-12
