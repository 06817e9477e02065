"""Both gradients of a variable-depth step in one call against the two calls."""
import pytest

from paper_2008_11607_gb300 import inputs
from tests.gpu_util import TOL, rel_l2, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("method,form,real", [("shared", "fp64", True), ("shared", "mixed", True),
                                              ("shared", "fp64", False), ("cg", "fp64", True)])
def test_backward_matches_adjoint_and_grad_depth(method, form, real):
    torch = torch_cuda()
    from paper_2008_11607_gb300 import rexi

    nx, ny = 40, 21
    H = torch.from_numpy(inputs.variable_depth(nx, ny, seed=3)).cuda()
    plan = rexi.Plan(nx, ny, depth=H, form=form)
    plan.set_krylov(rtol=1e-12)
    plan.set_krylov_method(method)
    dt = 10.0 / plan.rho
    x = to_dev(torch, inputs.white_real_state(nx, ny, seed=2))
    g = to_dev(torch, inputs.white_real_state(nx, ny, seed=4))
    gs, gd = plan.step_backward(x, g, dt, real_input=real)
    assert rel_l2(gs.cpu().numpy(), plan.step_adjoint(g, dt, real_input=real).cpu().numpy()) < TOL[form]
    assert rel_l2(gd.cpu().numpy(), plan.grad_depth(x, g, dt, real_input=real).cpu().numpy()) < 1e-12
    with pytest.raises(rexi.RexiError) as err:  # grad_in over the gradient it comes from
        rexi._check(plan._lib.rexi_step_backward(plan._h, x.data_ptr(), g.data_ptr(), g.data_ptr(), gd.data_ptr(), dt,
                                                 1e-10, 1, x.data_ptr() // 256 * 256, 1 << 20, 0), "backward")
    assert err.value.status == rexi.REXI_EINVAL


@pytest.mark.parametrize("method,real", [("cg", True), ("cg", False), ("shared", False)])
def test_an_adjoint_that_fails_adds_nothing_to_the_gradient(method, real):
    torch = torch_cuda()
    from paper_2008_11607_gb300 import rexi

    nx, ny = 40, 21
    H = torch.from_numpy(inputs.variable_depth(nx, ny, seed=3)).cuda()
    plan = rexi.Plan(nx, ny, depth=H)
    plan.set_krylov(rtol=1e-12, max_iters=3)
    plan.set_krylov_method(method)
    dt = 10.0 / plan.rho
    x = to_dev(torch, inputs.white_real_state(nx, ny, seed=2))
    g = to_dev(torch, inputs.white_real_state(nx, ny, seed=4))
    grad = torch.ones(ny, nx, dtype=torch.float64, device="cuda")
    with pytest.raises(rexi.RexiError) as err:
        plan.step_backward(x, g, dt, real_input=real, grad=grad)
    assert err.value.status == rexi.REXI_ENOCONV
    assert torch.equal(grad, torch.ones_like(grad))
