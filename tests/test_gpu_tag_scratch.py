"""The scratch that a geometry keeps for its refinement tags is part of the
device memory that it reports."""
import ctypes as C

import pytest
import torch

from paper_1809_03745_gb300 import workloads as W

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1809_03745_gb300 import ebpoisson as E


def _bytes(g):
    gi = E.GeomInfo()
    assert E.load().eb_geom_query(g._h, C.byref(gi)) == 0
    return gi.device_bytes


def test_device_bytes_count_the_kept_scratch():
    g = E.Geometry(W.pin_plane_3d(64))
    before = _bytes(g)
    field = torch.rand(3, 2, g.ncell, dtype=torch.float64, device="cuda")
    E.tag_cells(g, field)
    held = _bytes(g) - before
    assert 4 * g.ncell <= held <= 4 * g.ncell + 4096
    E.tag_cells(g, field)
    assert _bytes(g) - before == held
