"""Implicit 2-D steps in one launch (meshes up to 2^20 nodes): meshes of one,
few and more tiles than blocks, ragged tiles, restarts of the Krylov basis,
launches of 64 steps, a given first iterate, and the failure paths, against the
FP64 oracle's Newton roots."""
import numpy as np
import pytest
import torch

import oracle as O
import pf_inputs as G

pytestmark = pytest.mark.gpu


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b))


def solver(shape, model, dt, h=1.0, W=1.0):
    import paper_2601_06079_gb300 as pf
    s = pf.Solver(shape, h=h, model=model)
    s.set_params(W=W, kappa=0.7, mobility=1.1, dt=dt)
    return s, O.Problem(shape, h=h, W=W, kappa=0.7, mob=1.1)


@pytest.mark.parametrize("shape,h,restart", [((2, 2), 1.0, 30), ((5, 33), 1.0, 31),
                                             ((17, 31), (0.8, 1.3), 3), ((130, 65), 1.0, 30),
                                             ((301, 417), 1.0, 5)])
def test_ac_root(shape, h, restart):
    s, P = solver(shape, "ac", 0.5, h)
    U0 = G.ac_initial(4, shape, 0.2, 0.8)
    t = torch.from_numpy(U0).cuda()
    st = s.step_implicit(t, 1, newton_rtol=1e-6, gmres_rtol=1e-4, gmres_restart=restart)
    ref, info = P.newton(0.5, U0.astype(np.float64), abs_tol=1e-10, gmres_rtol=1e-8)
    assert st["converged"] and info["ok"]
    assert rel(t.cpu().numpy(), ref) <= 1e-5


@pytest.mark.parametrize("shape,restart", [((3, 3), 30), ((40, 70), 4), ((250, 331), 31)])
def test_ch_root(shape, restart):
    s, P = solver(shape, "ch", 0.05)
    c0 = G.ch_initial(5, shape)
    t = torch.from_numpy(c0).cuda()
    st = s.step_implicit(t, 1, newton_rtol=1e-7, gmres_rtol=1e-5, gmres_restart=restart)
    U, info = P.chsplit_newton(0.05, c0.astype(np.float64), abs_tol=1e-9)
    assert st["converged"] and info["ok"]
    assert rel(t.cpu().numpy(), U[0]) <= 1e-5


def test_more_steps_than_a_launch_equal_single_steps():
    s, _ = solver((33, 47), "ac", 0.25)
    a = torch.from_numpy(G.ac_initial(6, (33, 47), 0.3, 0.7)).cuda()
    b = a.clone()
    st = s.step_implicit(a, 70)
    n = sum(s.step_implicit(b, 1)["newton_iters"] for _ in range(70))
    assert st["converged"] and st["newton_iters"] == n
    assert torch.equal(a, b)


def test_root_as_guess_needs_no_iteration():
    s, _ = solver((64, 50), "ac", 0.5)
    U0 = torch.from_numpy(G.ac_initial(7, (64, 50), 0.2, 0.8)).cuda()
    root = U0.clone()
    s.step_implicit(root, 1, newton_rtol=1e-7, gmres_rtol=1e-5)
    t = U0.clone()
    st = s.step_implicit(t, 1, guess=root, newton_rtol=1e-5)
    assert st["newton_iters"] == 0 and torch.equal(t, root)


def test_failures_are_reported():
    import paper_2601_06079_gb300 as pf
    s, _ = solver((48, 48), "ac", 0.5)
    U0 = torch.from_numpy(G.ac_initial(8, (48, 48), 0.2, 0.8)).cuda()
    st = s.step_implicit(U0.clone(), 2, max_newton=1, newton_rtol=1e-7, check=False)
    assert st["status"] == pf._lib.PF_ERR_NOT_CONVERGED and not st["converged"]
    bad = U0.clone()
    bad[3, 5] = float("nan")
    keep = bad.clone()
    with pytest.raises(pf.PFError) as e:
        s.step_implicit(bad, 1)
    assert e.value.status == pf._lib.PF_ERR_NONFINITE
    assert torch.equal(torch.nan_to_num(bad, -1.0), torch.nan_to_num(keep, -1.0))
    assert s.step_implicit(U0, 1)["converged"]  # the context still works
