"""Implicit 2-D steps on both sides of the limit of the one-launch form: 2^20
nodes, counting idle nodes of the 32 x 16 tiles (a fifth more than the others),
against the FP64 oracle's Newton roots.  The meshes above it take the solver that
launches a kernel per vector operation, also with Krylov bases of more than 16
vectors (two launches of products, the widest update) and short cycles.

Bars: the residual is at most 1e-6 of U/dt.  Allen-Cahn at dt = 0.8: the
Jacobian is at least 1/dt - 1 = 0.25, so the root is off by at most 1e-6 * 1.25 /
0.25 = 5e-6 of U; Cahn-Hilliard likewise by a few 1e-6.  1e-5."""
import numpy as np
import pytest
import torch

import oracle as O
import pf_inputs as G

pytestmark = pytest.mark.gpu


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b))


def solver(shape, model, dt):
    import paper_2601_06079_gb300 as pf
    s = pf.Solver(shape, model=model)
    s.set_params(W=1.0, kappa=0.7, mobility=1.1 if model == "ch" else 1.0, dt=dt)
    return s, O.Problem(shape, W=1.0, kappa=0.7, mob=1.1 if model == "ch" else 1.0)


# below: 1024^2 and a thin mesh of 1,563 tiles; above: 2^20 nodes passed by a
# little (odd sizes), and by the tiles alone (1,875 tiles of 64 nodes in use)
@pytest.mark.parametrize("shape", [(1024, 1024), (2, 50000), (1025, 1031), (2, 60000)])
def test_ac_root(shape):
    s, P = solver(shape, "ac", 0.8)
    U0 = G.ac_initial(4, shape, 0.2, 0.8)
    t = torch.from_numpy(U0).cuda()
    st = s.step_implicit(t, 1, newton_rtol=1e-6, gmres_rtol=1e-5, gmres_restart=31)
    ref, info = P.newton(0.8, U0.astype(np.float64), abs_tol=1e-9, gmres_rtol=1e-6)
    assert st["converged"] and info["ok"]
    assert rel(t.cpu().numpy(), ref) <= 1e-5


@pytest.mark.parametrize("shape", [(1000, 1040), (1025, 1031), (3, 60001)])
def test_ch_root(shape):
    s, P = solver(shape, "ch", 0.3)
    c0 = G.ch_initial(5, shape)
    t = torch.from_numpy(c0).cuda()
    st = s.step_implicit(t, 1, newton_rtol=1e-6, gmres_rtol=1e-5, gmres_restart=31)
    U, info = P.chsplit_newton(0.3, c0.astype(np.float64), abs_tol=1e-8, gmres_rtol=1e-4)
    assert st["converged"] and info["ok"]
    assert rel(t.cpu().numpy(), U[0]) <= 1e-5


def test_short_cycles_above_the_limit():
    # restarts (a residual from a Jacobian product, the basis used again)
    s, P = solver((3, 60001), "ch", 0.3)
    c0 = G.ch_initial(6, (3, 60001))
    t = torch.from_numpy(c0).cuda()
    st = s.step_implicit(t, 1, newton_rtol=1e-6, gmres_rtol=1e-4, gmres_restart=5,
                         gmres_max_iters=2000)
    U, info = P.chsplit_newton(0.3, c0.astype(np.float64), abs_tol=1e-8, gmres_rtol=1e-4)
    assert st["converged"] and info["ok"]
    assert rel(t.cpu().numpy(), U[0]) <= 1e-5


@pytest.mark.parametrize("shape", [(3, 50001), (3, 60001)])
def test_first_newton_step_with_a_long_basis(shape):
    # one Newton step solved to 1e-6 in cycles of 31 vectors.  |G| is about 5 |U|
    # here; the eliminated Jacobian is at least 1/dt, and a residual of the mu row
    # enters the c row through M^-1 K (norm 8): dt (1 + 8) 5e-6 = 1.35e-5 of U.
    s, P = solver(shape, "ch", 0.3)
    c0 = G.ch_initial(7, shape)
    t = torch.from_numpy(c0).cuda()
    st = s.step_implicit(t, 1, max_newton=1, newton_rtol=1e-7, gmres_rtol=1e-6, gmres_restart=31,
                         gmres_max_iters=400, check=False)
    U, _ = P.chsplit_newton(0.3, c0.astype(np.float64), abs_tol=1e-12, max_newton=1)
    assert st["newton_iters"] == 1 and st["gmres_iters"] > 16
    assert rel(t.cpu().numpy(), U[0]) <= 2e-5
