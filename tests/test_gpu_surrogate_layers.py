"""The surrogate's element-wise layers and gradient sums on volumes of more than
one tile in every direction, unequal sides and an odd number of samples:
through the identity network, whose loss and gradients the reference gives to
rounding (bounds of the identity-network test)."""
import numpy as np
import pytest
import torch

import pf_inputs as G
from tests.test_gpu_conv import GRAD_REL_ID, _identity_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hist,stiff,shape", [(1, 0.3, (1, 8, 32, 64, 128)),
                                              (0, 0.7, (3, 8, 16, 64, 64))])
def test_loss_and_gradient(hist, stiff, shape):
    import paper_2601_06079_gb300 as pf
    from tests import _torch_unet as R
    s = pf.Surrogate(history=hist)
    s.params.copy_(_identity_params().float().cuda())
    u = torch.from_numpy(G.random_field(6, shape, 0.0, 1.0)).cuda()
    du = torch.from_numpy(G.random_field(7, shape)).cuda()
    x = torch.cat([u - 0.01 * k * du for k in range(hist + 1)], dim=1).contiguous()
    y = u + 0.012 * du
    xd = x.cpu().double()
    loss, g = s.loss_grad(x, y, stiff=stiff)
    p = R.bf16_weights(s.params.detach().cpu().double()).requires_grad_(True)
    if hist:
        h, sc = R.history_input(xd)
        so = R.output_scale(xd, sc)
        lr = R.loss_history(p, h.float().to(torch.bfloat16).double(), xd, y.cpu().double(), so,
                            stiff, bf16=True)
    else:
        out = R.forward(p, x.cpu().to(torch.bfloat16).double(), bf16=True)[:, :8]
        lr = (R.stiff_apply(out - (y.cpu().double() - xd), stiff) ** 2).mean()
    lr.backward()
    gr, gg = p.grad.numpy(), g.cpu().double().numpy()
    assert abs(loss - lr.item()) <= 1e-6 * lr.item()
    assert float(np.linalg.norm(gg - gr) / np.linalg.norm(gr)) <= GRAD_REL_ID
