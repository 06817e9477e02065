"""A step of many Chebyshev steps in one launch whose blocks give up waiting for
each other's edges (a limit of 0 polls: every wait gives up at once, and every
block returns): NaN outputs, gradients left as they were, and an error status
that the host reads."""
import pytest

from paper_2008_11607_gb300 import inputs
from tests.gpu_util import rel_l2, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


def _timeout(rexi, call):
    with pytest.raises(rexi.RexiError) as err:
        call()
    assert err.value.status == rexi.REXI_ETIMEOUT


@pytest.mark.parametrize("form", ["fp64", "mixed"])
@pytest.mark.parametrize("nx,ny", [(96, 80), (5, 70)])
def test_wait_that_runs_out(nx, ny, form):
    torch = torch_cuda()
    from paper_2008_11607_gb300 import rexi

    H = torch.from_numpy(inputs.variable_depth(nx, ny, seed=3)).cuda()
    plan = rexi.Plan(nx, ny, depth=H, form=form)
    plan.set_krylov(rtol=1e-12)
    plan.set_krylov_method("shared")
    dt = 10.0 / plan.rho
    x = to_dev(torch, inputs.white_real_state(nx, ny, seed=2))
    g = to_dev(torch, inputs.white_real_state(nx, ny, seed=4))
    ref = plan.step(x, dt)
    ref_gs, ref_gd = plan.step_backward(x, g, dt)

    plan.set_edge_polls(0)
    out = plan.step(x, dt)
    assert torch.isnan(out.real).all()
    _timeout(rexi, lambda: plan.step(x, dt))  # reported once, in the place of the next call's work
    grad = torch.ones(ny, nx, dtype=torch.float64, device="cuda")
    gs, _ = plan.step_backward(x, g, dt, grad=grad)
    assert torch.isnan(gs.real).all() and torch.equal(grad, torch.ones_like(grad))
    _timeout(rexi, lambda: plan.grad_depth(x, g, dt, grad=grad))
    plan.grad_depth(x, g, dt, grad=grad)
    assert torch.equal(grad, torch.ones_like(grad))
    _timeout(rexi, lambda: plan.step_adjoint(g, dt))
    host = x.cpu().pin_memory()
    _timeout(rexi, lambda: plan.step_host(host, torch.empty_like(host), dt))

    plan.set_edge_polls()
    assert rel_l2(plan.step(x, dt).cpu().numpy(), ref.cpu().numpy()) == 0.0
    gs, gd = plan.step_backward(x, g, dt, grad=grad)
    assert torch.equal(gs, ref_gs) and rel_l2((gd - 1.0).cpu().numpy(), ref_gd.cpu().numpy()) < 1e-12
    with pytest.raises(rexi.RexiError) as err:
        plan.set_edge_polls(-1)
    assert err.value.status == rexi.REXI_EINVAL
