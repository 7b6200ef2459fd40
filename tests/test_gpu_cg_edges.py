"""The library's CG where the residual reaches zero, and with the gathers of 8 and 16 coils, against the oracle."""
import numpy as np
import pytest

from gpu_helpers import host, make_case, rel, to_dev
from oracle import jacobian as jb
from oracle.nufft import KBNufft
from test_gpu_cg import TOL, _cg

pytestmark = pytest.mark.gpu


def _solve(shape, om, b, S, lam, iters, C, **opts):
    from paper_2111_02912_gb300 import Plan
    plan = Plan(shape, to_dev(np.ascontiguousarray(om)), max_coils=C, **opts)
    return host(plan.cg_normal(to_dev(b), lam, iters, to_dev(S)))


@pytest.mark.parametrize("iters", [1, 2, 5])
def test_zero_right_hand_side(iters):
    """x = 0 solves it: no step of the iteration may divide zero by zero."""
    shape, M, C = (24, 20), 700, 2
    case = make_case(shape, M, C, True, seed=700)
    assert not _solve(shape, case["omega"], np.zeros_like(case["x"]), case["smaps"], 3.0, iters, C).any()


@pytest.mark.parametrize("lam", [2.0, 3.0])   # 1 / lam exact: the residual is zero after one step; or not
def test_no_points_and_more_iterations_than_needed(lam):
    shape, C = (24, 20), 2
    case = make_case(shape, 1, C, True, seed=701)
    x = _solve(shape, case["omega"][:, :0], case["x"], case["smaps"], lam, 4, C)
    assert rel(x, case["x"] / lam) < 1e-6   # one rounding of each of b and 1 / lam, 2^-24, per step


@pytest.mark.parametrize("scale", [1.0, 1e-12])
def test_iterating_past_convergence(scale):
    """lam far above the spectrum: a digit or more per step, so that forty steps take the residual of
    scale * b below the smallest FP32 square; the converged image stays."""
    shape, M, C, lam = (24, 20), 700, 3, 100.0 * 700
    case = make_case(shape, M, C, True, seed=702)
    op, S = KBNufft(shape, case["omega"]), case["smaps"]
    F = lambda v: jb.sense_adjoint(op, jb.sense_forward(op, v, S), S) + lam * v
    b = (scale * case["x"]).astype(np.complex64)
    x = _solve(shape, case["omega"], b, S, lam, 40, C)
    assert np.isfinite(x.view(np.float32)).all()
    assert rel(x, _cg(F, b.astype(np.complex128), 12)) < TOL


def test_nan_in_the_right_hand_side_is_not_hidden():
    shape, M, C = (24, 20), 700, 2
    case = make_case(shape, M, C, True, seed=703)
    b = case["x"].copy()
    b[3, 4] = np.nan
    assert np.isnan(_solve(shape, case["omega"], b, case["smaps"], 3.0, 2, C)).any()


@pytest.mark.parametrize("shape,M,C", [
    ((40, 34), 900, 16), ((24, 20), 700, 20), ((24, 20), 700, 12),   # coil quads (one group, two); pairs
    ((40, 34), 900, 8), ((16, 14, 12), 900, 8), ((24, 20), 700, 33),   # whole lines in 2-D and 3-D; single coils
])
def test_gathers_into_the_sorted_order(shape, M, C):
    case = make_case(shape, M, C, True, seed=704)
    lam, iters = 0.5 * M, 4
    op, S = KBNufft(shape, case["omega"]), case["smaps"]
    F = lambda v: jb.sense_adjoint(op, jb.sense_forward(op, v, S), S) + lam * v
    x = _solve(shape, case["omega"], case["x"], S, lam, iters, C)
    assert rel(x, _cg(F, case["x"].astype(np.complex128), iters)) < TOL
