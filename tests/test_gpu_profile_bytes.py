"""The benchmark hook's bytes per launch are those that the split phases have to
move."""
import pytest
import torch

from paper_1809_03745_gb300 import workloads as W

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1809_03745_gb300 import ebpoisson as E


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("dim", [2, 3])
def test_bytes_of_the_split_phases(dim, precision):
    """Per fine cell, w bytes a word: a colour reads the other colour's x, its
    own b and flags and writes its own x; the residual + restriction after a
    black pass reads x, the red b and flags, and per coarse cell reads the flags
    and writes b; the prolongation reads and writes x, reads the flags, and per
    coarse cell reads x."""
    d = W.rod_plane_2d(128) if dim == 2 else W.pin_plane_3d(48, radius=0.13)
    P = E.Poisson(E.Geometry(d), precision=precision)
    n, w, c = P.geom.ncell, 4 if precision == "mixed" else 8, 2 ** dim
    for kernel, per in ((0, 1.5 * w + 0.5), (1, 1.5 * w + 0.5 + (w + 1) / c), (6, 2 * w + 1 + w / c)):
        ms, by = P.profile(kernel, reps=3)
        assert ms > 0.0 and by == pytest.approx(per * n)
