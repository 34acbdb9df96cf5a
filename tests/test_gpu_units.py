"""The solve does not depend on the units of its data: a problem whose data
are all multiplied by a power of two takes the same V-cycles to the same
potential, bit for bit, whatever the power (FP32 holds neither the data nor
the products of their residuals at most of these), and an initial guess that
is many orders of magnitude away from the solution is corrected."""
import copy

import numpy as np
import pytest
import torch

from paper_1809_03745_gb300 import workloads as W

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1809_03745_gb300 import ebpoisson as E


def _problem(dim):
    d = W.rod_plane_2d(120, dielectric=True, half_width=0.08, slab_y=0.2 + 0.3 / 120) if dim == 2 else \
        W.pin_plane_3d(40, radius=0.13, disk_t=3.3 / 40)
    rng = np.random.default_rng(17)
    n = W.ncells(d)
    S = np.zeros((2, n))
    S[0] = rng.uniform(-50, 100, n)
    return d, S, rng.uniform(-1, 1, n)


def _scaled(d, S, sig, f):
    d = copy.deepcopy(d)
    d["electrodes"] = [(r, v * f) for r, v in d["electrodes"]]
    d["phi_E"] *= f
    d["phi_wall"] = [v * f for v in d["phi_wall"]]
    return d, S * f, sig * f


def _solve(d, S, sig, phi=None, **kw):
    P = E.Poisson(E.Geometry(d), precision="mixed", tol=1e-12, max_cycles=400, **kw)
    phi, info = P.solve(torch.from_numpy(S), torch.from_numpy(sig), phi)
    assert info["status"] == 0, info
    return phi, info


@pytest.mark.parametrize("e", [-400, -83, 59, 83, 400])
@pytest.mark.parametrize("dim", [2, 3])
def test_scaled_data_give_the_scaled_solution(dim, e):
    d, S, sig = _problem(dim)
    want, iw = _solve(d, S, sig)
    f = 2.0 ** e
    got, ig = _solve(*_scaled(d, S, sig, f))
    assert ig["vcycles"] == iw["vcycles"], (ig, iw)
    assert torch.equal(got, want * f)


@pytest.mark.parametrize("exp", [-30, 30])
@pytest.mark.parametrize("dim", [2, 3])
def test_guess_far_from_the_solution(dim, exp):
    """Data of size 1 and a guess of size 1e30; and data of size 1e-30 with a
    guess of size 1: the residual starts 30 orders above max|b|."""
    d, S, sig = _problem(dim)
    want, _ = _solve(d, S, sig)
    f = 1.0 if exp > 0 else 2.0 ** -100
    gen = torch.Generator(device="cuda").manual_seed(3)
    phi = torch.randn(2, W.ncells(d), dtype=torch.float64, device="cuda", generator=gen)
    got, _ = _solve(*_scaled(d, S, sig, f), phi=phi * 10.0 ** max(exp, 0))
    # 1e-12 of max|b| holds phi to 1e-9, as in every parity case
    assert (got - want * f).abs().max() <= 1e-9 * (want * f).abs().max()


def test_batched_steps_equal_the_single_solve_at_any_unit():
    """The server resumes a solve launch by launch: the same iterates."""
    d, S, sig = _problem(2)
    for f in (1.0, 2.0 ** 90):
        q = _scaled(d, S, sig, f)
        want, iw = _solve(*q)
        srv = E.Server(max_slots=2, step_iters=1, tol=1e-12, max_cycles=400)
        try:
            phi, info = srv.wait(srv.submit(*q), 120.0)
        finally:
            srv.close()
        assert info["status"] == 0 and info["vcycles"] == iw["vcycles"]
        assert np.array_equal(phi, want.cpu().numpy())
