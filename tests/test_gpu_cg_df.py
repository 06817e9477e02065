"""Per-term CG of the FP64 form where its iterations run in double-float and are
checked in FP64 (rtol well above kappa 2^-48), against the sparse oracle, and
the calls that go on to the FP64 iterations.  Error bound as for the FP64
iterations (error_bound of tests/test_gpu_krylov.py)."""
import numpy as np
import pytest

from oracle import operator as O
from oracle import rexi as R
from paper_2008_11607_gb300 import inputs
from tests.gpu_util import rel_l2, to_dev, torch_cuda
from tests.test_gpu_krylov import error_bound, krylov_plan

pytestmark = pytest.mark.gpu
RTOL = 1e-10


@pytest.mark.parametrize("nx,ny,real", [(3, 3, True), (32, 16, False), (33, 17, True), (31, 34, False), (70, 5, True)])
def test_step_and_adjoint_at_tile_edges(nx, ny, real):
    torch = torch_cuda()
    phys = dict(Lx=1.3, Ly=0.8, g=1.4, f=0.7) if nx % 2 else {}
    H = inputs.variable_depth(nx, ny, seed=5)
    plan = krylov_plan(torch, nx, ny, H, rtol=RTOL, batch=17, **phys)
    dt = 5.0 / plan.rho
    st = inputs.complex_random_state(nx, ny, seed=6)
    if real:
        st = st.real.astype(np.complex128)
    got, info = plan.step(to_dev(torch, st), dt, real_input=real, want_info=True)
    assert info.krylov_unconverged == 0 and 0.0 < info.krylov_max_rel_res <= RTOL
    A = O.cgrid_operator(nx, ny, H=H, **phys)
    tol = error_bound(info.M, RTOL, H, phys.get("g", 1.0), real)
    ref = R.rexii_apply_sparse(A, st.ravel(), dt, 0.5, info.M, real_input=real).reshape(st.shape)
    assert rel_l2(got.cpu().numpy(), ref) < tol
    adj = plan.step_adjoint(to_dev(torch, st), dt, real_input=real).cpu().numpy()
    refa = np.conj(R.rexii_apply_sparse(A.T.tocsr(), np.conj(st).ravel(), dt, 0.5, info.M, real_input=real))
    assert rel_l2(adj.ravel(), refa) < tol


def test_values_beyond_single_precision_and_the_iteration_cap():
    from paper_2008_11607_gb300 import rexi

    torch = torch_cuda()
    nx, ny = 20, 18
    H = inputs.variable_depth(nx, ny, seed=5)
    plan = krylov_plan(torch, nx, ny, H, rtol=RTOL)
    dt = 8.0 / plan.rho
    st = inputs.kminus3_field(nx, ny, seed=6)
    ref, info = plan.step(to_dev(torch, st), dt, want_info=True)
    tol = 2.0 * error_bound(info.M, RTOL, H)
    for scale in (2.0 ** -200, 2.0 ** 200):  # the FP64 iterations
        got = plan.step(to_dev(torch, st * scale), dt).cpu().numpy() / scale
        assert rel_l2(got, ref.cpu().numpy()) < tol
    assert torch.count_nonzero(plan.step(torch.zeros_like(ref), dt)).item() == 0
    plan.set_krylov(rtol=RTOL, max_iters=3, term_batch=8)
    with pytest.raises(rexi.RexiError) as err:
        plan.step(to_dev(torch, st), dt)
    assert err.value.status == rexi.REXI_ENOCONV


def test_iteration_cap_in_double_float_leaves_the_fp64_iterations():
    """Terms that reach the cap in double-float have the FP64 iterations, under the same cap,
    before the call gives up: the launches of a call that runs only those (an rtol that
    double-float cannot reach) come on top of the double-float ones."""
    from paper_2008_11607_gb300 import rexi

    torch = torch_cuda()
    nx, ny = 20, 18
    plan = krylov_plan(torch, nx, ny, inputs.variable_depth(nx, ny, seed=5), rtol=RTOL)
    dt = 8.0 / plan.rho
    x = to_dev(torch, inputs.kminus3_field(nx, ny, seed=6))
    launches = {}
    for rtol in (RTOL, 1e-14):
        plan.set_krylov(rtol=rtol, max_iters=3, term_batch=8)
        plan.set_profiling(True)
        with pytest.raises(rexi.RexiError) as err:
            plan.step(x, dt)
        assert err.value.status == rexi.REXI_ENOCONV
        launches[rtol] = plan.read_profile()[2]
    assert launches[RTOL] >= 2 * launches[1e-14]


def test_double_float_iterations_run_and_the_check_rejects():
    """Ordinary values take the double-float iterations alone.  Values beyond FP32's exponents leave
    them at x = 0, which the FP64 check rejects: those launches come on top of the FP64 iterations."""
    torch = torch_cuda()
    nx, ny = 20, 18
    plan = krylov_plan(torch, nx, ny, inputs.variable_depth(nx, ny, seed=5), rtol=RTOL)
    dt = 8.0 / plan.rho
    st = inputs.kminus3_field(nx, ny, seed=6)
    launches = []
    for scale in (1.0, 2.0 ** -200):
        plan.set_profiling(True)
        _, info = plan.step(to_dev(torch, st * scale), dt, want_info=True)
        launches.append(plan.read_profile()[2])
        assert info.krylov_unconverged == 0 and info.krylov_max_rel_res <= RTOL
    assert launches[0] < launches[1]
