"""Conjugate gradients with the sums finished inside the operator and update
launches: meshes without interior nodes, with one and with several blocks, and
lengths that are no multiple of four, solved into aligned and unaligned
buffers, against the oracle's solution."""
import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(2, 2, 2), (3, 3, 3), (5, 7, 9), (17, 6, 18), (4, 18, 35)])
@pytest.mark.parametrize("offset", [0, 1])
def test_solution_matches_oracle(shape, offset):
    import paper_2601_06079_gb300 as pf
    h, m, l, a = (1.0, 1.2, 0.9), 0.01, 0.5, 3.0
    ref, ok, _ = O.Elastic(shape, h).solve(22.5, 0.3, m, l, a, rtol=1e-12)
    assert ok
    el = pf.Elastic(shape, h, E=22.5, nu=0.3, m=m, l=l, a=a)
    n = 3 * int(np.prod(shape))
    u = torch.zeros(n + offset, device="cuda")[offset:].view(3, *shape)
    el.solve(u=u, rtol=1e-7)
    assert el.stats.converged == 1
    # the bar of the existing solution test
    err = u.cpu().numpy().astype(np.float64) - ref
    assert np.linalg.norm(err) <= 1e-5 * np.linalg.norm(ref)
