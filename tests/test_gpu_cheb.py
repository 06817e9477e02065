"""The Chebyshev form of the shared-Krylov method (cheb.cu) at the sizes where
its tiles and halos can go wrong, against the sparse oracle, and the calls
that it leaves to the Lanczos form.

Tolerance as for the Lanczos form: the error bound rtol in the energy norm,
converted by sqrt(max w / min w), times 10; double-float arithmetic adds
TOL["mixed"]."""
import math

import numpy as np
import pytest

from oracle import adjoint as AD
from oracle import operator as O
from oracle import rexi as R
from paper_2008_11607_gb300 import inputs
from tests.gpu_util import TOL, rel_l2, to_dev, torch_cuda

pytestmark = pytest.mark.gpu
RTOL = 1e-12


def _plan(torch, nx, ny, H, form, rtol=RTOL, **phys):
    from paper_2008_11607_gb300 import rexi

    plan = rexi.Plan(nx, ny, depth=torch.from_numpy(np.ascontiguousarray(H)).cuda(), form=form, **phys)
    plan.set_krylov(rtol=rtol)
    plan.set_krylov_method("shared")
    return plan


def _tol(form, H, g=1.0):
    w = np.concatenate([g / np.ravel(H), np.ones(1)])
    return max(TOL[form], 10 * RTOL * math.sqrt(w.max() / w.min()))


# one tile exactly, one short of it, one past it, several with ragged edges,
# the smallest grid, and strips narrower than a tile
@pytest.mark.parametrize("nx,ny,taurho", [(3, 3, 4.0), (32, 16, 6.0), (31, 15, 6.0), (33, 17, 6.0), (65, 34, 4.0),
                                          (5, 70, 5.0), (70, 3, 30.0)])
def test_step_adjoint_gradient_at_tile_edges(nx, ny, taurho):
    """Real input against the real part of the complex oracle (the matrix r(dt A) is real)."""
    torch = torch_cuda()
    phys = dict(Lx=1.3, Ly=0.8, g=1.4, f=0.7) if nx % 2 else {}
    H = inputs.variable_depth(nx, ny, seed=5)
    st = inputs.complex_random_state(nx, ny, seed=6)
    G = inputs.complex_random_state(nx, ny, seed=7).real.astype(np.complex128)
    re = st.real.astype(np.complex128)
    A = O.cgrid_operator(nx, ny, H=H, **phys)
    ref = None
    for form in ("fp64", "mixed"):
        plan = _plan(torch, nx, ny, H, form, **phys)
        dt = taurho / plan.rho
        tol = _tol(form, H, phys.get("g", 1.0))
        got, info = plan.step(to_dev(torch, st), dt, real_input=False, want_info=True)
        assert info.krylov_max_rel_res <= RTOL
        if ref is None:
            ref = R.rexii_apply_sparse(A, st.ravel(), dt, 0.5, info.M, real_input=False).reshape(st.shape)
            refa = np.conj(R.rexii_apply_sparse(A.T.tocsr(), np.conj(st).ravel(), dt, 0.5, info.M, real_input=False))
            refa = refa.reshape(st.shape)
            refg = AD.grad_depth_sparse(nx, ny, H, re.ravel(), G.ravel(), dt, 0.5, info.M, **phys)
        assert rel_l2(got.cpu().numpy(), ref) < tol
        assert rel_l2(plan.step(to_dev(torch, re), dt).cpu().numpy(), ref.real) < tol
        assert rel_l2(plan.step_adjoint(to_dev(torch, st), dt, real_input=False).cpu().numpy(), refa) < tol
        assert rel_l2(plan.step_adjoint(to_dev(torch, re), dt).cpu().numpy(), refa.real) < tol
        start = torch.ones(ny, nx, dtype=torch.float64, device="cuda")  # the call adds to what is there
        grad = plan.grad_depth(to_dev(torch, re), to_dev(torch, G), dt, grad=start).cpu().numpy() - 1.0
        assert rel_l2(grad, refg) < max(1e-9, tol)


@pytest.mark.parametrize("form", ["fp64", "mixed"])
@pytest.mark.parametrize("nx,ny,real", [(1001, 650, True), (507, 495, False), (640, 343, True)])
def test_grids_beyond_shared_memory_match_fourier(nx, ny, real, form):
    """Ragged grids that take one launch per step (the last: the largest that the
    tiles hold, nearly), with H = 1 against the Fourier path."""
    torch = torch_cuda()
    from paper_2008_11607_gb300 import rexi

    st = inputs.complex_random_state(nx, ny, seed=3)
    if real:
        st = st.real.astype(np.complex128)
    plan = _plan(torch, nx, ny, np.ones((ny, nx)), form)
    dt = 20.0 / plan.rho
    x = to_dev(torch, st)
    got = plan.step(x, dt, real_input=real)
    ref = rexi.Plan(nx, ny).step(x, dt, real_input=real)
    assert rel_l2(got.cpu().numpy(), ref.cpu().numpy()) < _tol(form, np.ones(1))


@pytest.mark.parametrize("form", ["fp64", "mixed"])
def test_gradient_beyond_shared_memory_matches_lanczos(form):
    """The depth gradient at 701 x 650 (one launch per step) against the two-sided
    Lanczos form, which a bound below 1e-13 selects; the tolerance of the
    gradient's oracle tests."""
    torch = torch_cuda()
    nx, ny = 701, 650
    H = inputs.variable_depth(nx, ny, seed=5)
    x = to_dev(torch, inputs.kminus3_field(nx, ny, seed=6))
    G = to_dev(torch, inputs.kminus3_field(nx, ny, seed=7))
    plan = _plan(torch, nx, ny, H, form)
    dt = 10.0 / plan.rho
    got = plan.grad_depth(x, G, dt).cpu().numpy()
    ref = _plan(torch, nx, ny, H, "fp64", rtol=9e-14).grad_depth(x, G, dt).cpu().numpy()
    assert rel_l2(got, ref) < 1e-9


@pytest.mark.parametrize("form", ["fp64", "mixed"])
def test_options_and_calls_left_to_the_lanczos_form(form):
    """A spacing h whose alias the expansion would have to resolve, and values
    outside the exponents that the expansion takes; and a rho set above the
    operator's (more terms, the same interval): against the oracle."""
    torch = torch_cuda()
    nx, ny = 24, 20
    H = inputs.variable_depth(nx, ny, seed=5)
    st = inputs.kminus3_field(nx, ny, seed=6)
    A = O.cgrid_operator(nx, ny, H=H)
    tol = _tol(form, H)
    wide = _plan(torch, nx, ny, H, form, h=1.0)
    dt = 20.0 / wide.rho
    got, info = wide.step(to_dev(torch, st), dt, want_info=True)
    assert rel_l2(got.cpu().numpy(), R.rexii_apply_sparse(A, st.ravel(), dt, 1.0, info.M).reshape(st.shape)) < tol
    plan = _plan(torch, nx, ny, H, form)
    ref, info = plan.step(to_dev(torch, st), dt, want_info=True)
    for scale in (2.0 ** -80, 2.0 ** 80):
        got = plan.step(to_dev(torch, st * scale), dt).cpu().numpy() / scale
        assert rel_l2(got, ref.cpu().numpy()) < tol
    plan.set_rho(2.0 * plan.rho)
    got, info = plan.step(to_dev(torch, st), dt, want_info=True)
    assert rel_l2(got.cpu().numpy(), R.rexii_apply_sparse(A, st.ravel(), dt, 0.5, info.M).reshape(st.shape)) < tol


def test_declined_input_stops_the_steps():
    """Input that is left to the Lanczos form (values outside double-float's exponents), on a grid with
    one launch per step: no more than 16 Chebyshev steps, and six launches around them, come on top of
    the Lanczos form's launches (alone under a cap one step below the Chebyshev degree)."""
    torch = torch_cuda()
    nx, ny = 701, 650
    plan = _plan(torch, nx, ny, inputs.variable_depth(nx, ny, seed=5), "mixed", rtol=1e-8)
    dt = 200.0 / plan.rho
    x = to_dev(torch, inputs.kminus3_field(nx, ny, seed=6))
    _, info = plan.step(x, dt, want_info=True)
    launches = []
    for cap in (20000, info.krylov_iters - 1):
        plan.set_krylov(rtol=1e-8, max_iters=cap)
        plan.set_profiling(True)
        assert torch.isfinite(plan.step(x * 2.0 ** -80, dt).real).all()
        launches.append(plan.read_profile()[2])
    assert launches[1] < launches[0] <= launches[1] + 22


# tiles of one launch; a grid beyond shared memory; thin complex ones (two sets) whose
# tiles' edges are too long, narrower than the tile of the other kernel
@pytest.mark.parametrize("form", ["fp64", "mixed"])
@pytest.mark.parametrize("nx,ny,real,tiles", [(33, 17, True, True), (70, 3, False, True), (96, 80, True, True),
                                              (701, 650, True, False), (16384, 11, False, False),
                                              (5, 16384, False, False)])
def test_which_kernel_a_grid_takes(nx, ny, real, tiles, form):
    """The launch count tells one launch for many steps from one launch per step; the
    latter against the Lanczos form, which a bound below 1e-13 selects."""
    torch = torch_cuda()
    H = inputs.variable_depth(nx, ny, seed=5)
    st = inputs.complex_random_state(nx, ny, seed=6)
    x = to_dev(torch, st.real if real else st)
    plan = _plan(torch, nx, ny, H, form)
    dt = 8.0 / plan.rho

    def launches(call):
        plan.set_profiling(True)
        out = call()
        return out, plan.read_profile()[2]

    (got, info), n = launches(lambda: plan.step(x, dt, real_input=real, want_info=True))
    K = info.krylov_iters
    assert n <= 6 if tiles else K <= n <= K + 5
    if real:
        g = to_dev(torch, inputs.complex_random_state(nx, ny, seed=7).real)
        (gs, gd), n = launches(lambda: plan.step_backward(x, g, dt))
        assert n <= 12 if tiles else n >= 2 * K
    if not tiles:
        other = _plan(torch, nx, ny, H, "fp64", rtol=9e-14)
        tol = _tol(form, H)
        assert rel_l2(got.cpu().numpy(), other.step(x, dt, real_input=real).cpu().numpy()) < tol
        if real:
            ref_gs, ref_gd = other.step_backward(x, g, dt)
            assert rel_l2(gs.cpu().numpy(), ref_gs.cpu().numpy()) < tol
            assert rel_l2(gd.cpu().numpy(), ref_gd.cpu().numpy()) < max(1e-9, tol)
