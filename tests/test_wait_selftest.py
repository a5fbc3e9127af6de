"""The bounded waits between blocks of one launch (explicit trajectories held on
chip, implicit 2-D steps in one launch): with a block missing they run out, the
call reports it and the context stays usable."""
import pytest
import torch

import pf_inputs as G


def test_arguments_are_checked_on_the_host():
    from paper_2601_06079_gb300 import _lib
    _lib.lib()
    par = _lib.pf_params(1.0, 0.5, 1.0, 1e-3, 1.0, 1.0, 1.5, 0.5, None, 150.0)
    st, ctx, ws = _lib.pf_create_mesh(2, [400, 300], [1.0, 1.0], _lib.PF_MODEL_AC, 1, 0)
    assert st == 0
    assert _lib.pf_wait_selftest(ctx, 0x1000, 20, 1000, 0) == _lib.PF_ERR_STATE
    st, ex = _lib.pf_explicit_workspace(ctx)
    assert _lib.pf_bind_workspace(ctx, 0x100000, ex) == 0
    assert _lib.pf_set_params(ctx, par) == 0
    for bad in ((0, 20, 1000), (0x1000, 7, 1000), (0x1000, 20, 0), (0x1000, 1 << 40, 1000)):
        assert _lib.pf_wait_selftest(ctx, *bad, 0) == _lib.PF_ERR_ARG
    assert _lib.pf_wait_selftest(ctx, 0x1000, 20, 1000, 1) == _lib.PF_ERR_STATE  # explicit only
    _lib.pf_destroy(ctx)
    for model, nodes in ((_lib.PF_MODEL_COUPLED, [64, 64]), (_lib.PF_MODEL_AC, [4, 4]),
                         (_lib.PF_MODEL_AC, [8192, 8192])):
        nf = 2 if model == _lib.PF_MODEL_COUPLED else 1
        st, ctx, ws = _lib.pf_create_mesh(2, nodes, [1.0, 1.0], model, nf, 0)
        assert st == 0 and _lib.pf_bind_workspace(ctx, 0x100000, ws) == 0
        assert _lib.pf_set_params(ctx, par) == 0
        for implicit in (0, 1):
            assert _lib.pf_wait_selftest(ctx, 0x1000, 20, 1000, implicit) == _lib.PF_ERR_ARG
        _lib.pf_destroy(ctx)


@pytest.mark.gpu
@pytest.mark.parametrize("model", ["ac", "ch"])
def test_onchip_wait_runs_out_and_is_reported(model):
    import paper_2601_06079_gb300 as pf
    from paper_2601_06079_gb300 import _lib
    s = pf.Solver((300, 310), model=model)
    s.set_params(W=1.0, kappa=0.5, mobility=1.0, dt=1e-3)
    u0 = torch.from_numpy(G.ch_initial(1, (300, 310))).cuda()
    u = u0.clone()
    assert _lib.pf_wait_selftest(s._ctx, u.data_ptr(), 40, 20_000_000, 0) == _lib.PF_ERR_TIMEOUT
    assert torch.isnan(u).any()
    with pytest.raises(pf.PFError) as e:
        s.energy(u0)
    assert e.value.status == _lib.PF_ERR_TIMEOUT
    a, b = u0.clone(), u0.clone()
    s.step_explicit(a, 40)
    s.energy(a)
    s.set_form("fused_stream")
    s.step_explicit(b, 40)
    assert torch.equal(a, b)


@pytest.mark.gpu
@pytest.mark.parametrize("model", ["ac", "ch"])
def test_implicit_wait_runs_out_and_is_reported(model):
    import paper_2601_06079_gb300 as pf
    from paper_2601_06079_gb300 import _lib
    s = pf.Solver((200, 210), model=model)
    s.set_params(W=1.0, kappa=0.7, mobility=1.0, dt=0.25)
    u0 = torch.from_numpy(G.ch_initial(2, (200, 210))).cuda()
    ref = u0.clone()
    assert s.step_implicit(ref, 2)["converged"]
    u = u0.clone()
    assert _lib.pf_wait_selftest(s._ctx, u.data_ptr(), 8, 20_000_000, 1) == _lib.PF_ERR_TIMEOUT
    u = u0.clone()
    assert s.step_implicit(u, 2)["converged"]
    assert torch.equal(u, ref)
