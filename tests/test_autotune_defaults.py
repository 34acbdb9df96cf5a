"""With nothing cached the autotuner leaves the schedule to the library, which
chooses by the path that runs (host logic, a stand-in for the solver)."""
from types import SimpleNamespace

import pytest

from paper_1809_03745_gb300 import autotune as A
from paper_1809_03745_gb300 import ebpoisson as E


@pytest.mark.parametrize("dim,own", [(2, (2, 2, 2)), (3, (3, 3, 2))])
def test_solver_without_a_cached_schedule_takes_the_library_default(dim, own, monkeypatch):
    got = {}
    monkeypatch.setattr(E, "Poisson", lambda geom, **kw: got.update(kw))
    g = SimpleNamespace(dim=dim, ncell=64 ** dim, info=dict(n_phase=1))
    t = A.Autotuner(None)
    t.solver(g, launch_mode=2)
    assert got["nu1"] == got["nu2"] == -1 and got["inner_cycles"] == 2 and got["launch_mode"] == 2
    assert t.schedule(g) == own  # what that is on the default path
    t.table[A.size_class(dim, g.ncell, 1, "mixed")] = {"schedule": [4, 1, 3], "trials": []}
    t.solver(g)
    assert (got["nu1"], got["nu2"], got["inner_cycles"]) == (4, 1, 3)
    assert t.schedule(g) == (4, 1, 3)
