"""The mobility-field step and its reverse sweep at strip and band edges (60
columns, 4 rows), odd widths, segments shorter and longer than the trajectory,
and unequal spacings, against the oracle's step and adjoint."""
import numpy as np
import pytest
import torch

import oracle as O
import pf_inputs as G

pytestmark = pytest.mark.gpu


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b))


@pytest.mark.parametrize("shape,h,ckpt", [((3, 3), 1.0, 5), ((4, 60), 1.0, 12),
                                          ((9, 61), (0.9, 1.2), 1), ((5, 121), 1.0, 30),
                                          ((62, 59), (1.1, 0.8), 8)])
def test_step_and_adjoint(shape, h, ckpt):
    import paper_2601_06079_gb300 as pf
    n = 24
    c0, mob = G.ch_initial(3, shape, amp=0.2), G.random_field(4, shape, 0.5, 1.5)
    target = G.ch_initial(5, shape, amp=0.1)
    s = pf.Solver(shape, h=h, model="ch")
    s.set_params(W=1.2, kappa=0.5, mobility=0.9, dt=1e-3, mobility_field=torch.from_numpy(mob))
    P = O.Problem(shape, h=h, W=1.2, kappa=0.5, mob=0.9, mob_field=mob.astype(np.float64))
    t = torch.from_numpy(c0).cuda()
    s.step_explicit(t, n)
    assert rel(t.cpu().numpy(), P.ch_explicit(c0, 1e-3, n)) <= 1e-6
    loss, g = s.adjoint(torch.from_numpy(c0).cuda(), torch.from_numpy(target).cuda(), n, ckpt,
                        want_state=True)
    rloss, ref = P.ch_adjoint(c0, target, 1e-3, n)
    assert abs(loss - rloss) <= 1e-6 * abs(rloss)
    # gradient bar of the calibration tests
    for k in ("kappa", "W", "M"):
        assert abs(g[k] - ref[k]) <= 1e-4 * abs(ref[k]), k
    assert rel(g["mobility_field"].cpu().numpy(), ref["mob_field"]) <= 1e-4
    assert rel(g["c0"].cpu().numpy(), ref["c0"]) <= 1e-5
