"""Real input on grids of odd nx (pairs of rows share one transform) against the
same step on the full complex spectrum, forward and adjoint."""
import numpy as np
import pytest

from paper_2008_11607_gb300 import inputs
from tests.gpu_util import TOL, rel_l2, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["fp64", "mixed"])
@pytest.mark.parametrize("nx,ny", [(3, 2), (3, 5), (33, 20), (375, 7), (99, 31), (1155, 64)])
def test_odd_rows_match_full_spectrum(nx, ny, form):
    torch = torch_cuda()
    from paper_2008_11607_gb300 import rexi

    plan = rexi.Plan(nx, ny, form=form)
    dt = 30.0 / plan.rho
    x = to_dev(torch, inputs.white_real_state(nx, ny, seed=2))
    for step in (plan.step, plan.step_adjoint):
        got, ref = step(x, dt, real_input=True).cpu().numpy(), step(x, dt, real_input=False).cpu().numpy()
        assert np.all(got.imag == 0)
        assert rel_l2(got, ref.real) < TOL[form]
