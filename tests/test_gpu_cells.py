"""The pole sum by local expansion against the direct sum per orbit: the step is
linear in the terms, and a slice of a few terms takes the direct sum, so the
slices of one term range must add up to the one call that takes the cells.

Tolerance: each slice rounds its transforms at 8 u log2(nx ny) of its result
(u = 2^-53, or 2^-48 in double-float arithmetic), and the slices' results sum to
at most about 50 in magnitude (the tails 1 / y of the terms), so the sum of the
slices is within 50 * 8 * 17 u of the whole: 8e-13 and 2.4e-11."""
import numpy as np
import pytest

from paper_2008_11607_gb300 import inputs
from tests.gpu_util import rel_l2, to_dev, torch_cuda

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "mixed": 2.5e-11}

# nx, ny, tau rho, h, symbol, coefficients, shift, real input, term range
CASES = {
    "real_two_level": (256, 250, 400.0, 0.5, "cgrid", "rexii", "none", True, (0, -1)),
    "complex_odd_grid": (255, 243, 150.0, 0.5, "cgrid", "rexii", "none", False, (0, -1)),
    "h_off_the_split_grid": (256, 200, 150.0, 0.3, "cgrid", "rexii", "none", True, (0, -1)),
    "gap_in_the_terms": (256, 250, 300.0, 0.5, "cgrid", "rexii", "none", True, (37, 500)),
    "outer_terms": (256, 250, 300.0, 0.5, "cgrid", "rexii", "none", False, (500, -1)),
    "spectral": (200, 256, 200.0, 0.5, "spectral", "rexii", "none", False, (0, -1)),
    "original_rexi": (256, 256, 60.0, 0.2, "cgrid", "rexi", "none", True, (0, -1)),
    "signed_range": (250, 256, 300.0, 0.5, "schrodinger", "rexie", "midpoint", False, (0, -1)),
    "negative_range": (200, 243, 200.0, 0.5, "schrodinger", "rexii", "none", False, (0, -1)),
}


@pytest.mark.parametrize("form", ["fp64", "mixed"])
@pytest.mark.parametrize("case", sorted(CASES))
def test_cells_against_direct_slices(case, form):
    torch = torch_cuda()
    from paper_2008_11607_gb300 import rexi

    nx, ny, tau_rho, h, symbol, coefs, shift, real, (tb, te) = CASES[case]
    plan = rexi.Plan(nx, ny, form=form, h=h)
    plan.set_symbol(symbol)
    plan.set_coefficients(coefs)
    plan.set_shift(shift)
    dt = tau_rho / plan.rho
    x = to_dev(torch, inputs.white_real_state(nx, ny, 3) if real else inputs.complex_random_state(nx, ny, 3))
    ws = plan.workspace(dt, real_input=real)

    def step(lo, hi):
        plan.set_profiling(True)
        out = plan.step(x, dt, real_input=real, workspace=ws, terms=(lo, hi))
        return out, plan.read_profile()[2]

    whole, launches = step(tb, te)
    last = plan.step(x, dt, real_input=real, workspace=ws, want_info=True)[1].N + 1 if te < 0 else te
    total = torch.zeros_like(whole)
    for lo in range(tb, last, 8):
        part, direct = step(lo, min(lo + 8, last))
        assert direct < launches  # a few terms: summed directly
        total += part
    assert rel_l2(whole.cpu().numpy(), total.cpu().numpy()) < TOL[form]
    # dt = 0: one cell, every wavenumber at x = 0
    still = plan.step(x, 0.0, real_input=real, workspace=ws).cpu().numpy()
    if coefs != "rexi":
        assert rel_l2(still, np.asarray(x.cpu())) < 1e-10


@pytest.mark.parametrize("h", [1.0, 2.0])
def test_wide_spacing_against_fp64(h):
    """Cells of half-width 1 and 2: the mixed form against the FP64 form, within the rounding of both
    term sums and of the transforms (the error model of tests/gpu_util.py)."""
    torch = torch_cuda()
    from paper_2008_11607_gb300 import rexi
    from tests.gpu_util import fft_rounding_bound, pole_rounding_bound

    nx, ny, tau_rho = 256, 250, 200.0
    x = to_dev(torch, inputs.white_real_state(nx, ny, 3))
    out, launches, tol = {}, {}, 0.0
    for form in ("fp64", "mixed"):
        plan = rexi.Plan(nx, ny, form=form, h=h)
        dt = tau_rho / plan.rho
        plan.set_profiling(True)
        out[form], info = plan.step(x, dt, want_info=True)
        launches[form] = plan.read_profile()[2]
        plan.step(x, dt, terms=(0, 8))
        assert plan.read_profile()[2] < launches[form]  # the whole sum took the cells
        tol += pole_rounding_bound(form, tau_rho, h, info.M) + fft_rounding_bound(form, nx, ny)
    assert rel_l2(out["mixed"].cpu().numpy(), out["fp64"].cpu().numpy()) < tol
