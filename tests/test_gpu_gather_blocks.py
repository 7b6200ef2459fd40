"""Single-coil gathers in both block forms (which one depends on dimension, J, product and coil count), against the oracle."""
import pytest

from gpu_helpers import host, make_case, rel, to_dev
from oracle import jacobian as jb
from oracle.nufft import KBNufft

pytestmark = pytest.mark.gpu

TOL = 1e-5   # FP32 rounding of transforms and taps: the tolerance of the parity tests


@pytest.mark.parametrize("shape,J", [((60,), 6), ((60,), 8), ((24, 20), 6), ((24, 20), 7)] + [((12, 14, 12), J) for J in (4, 5, 6, 7, 8)])
@pytest.mark.parametrize("C", [1, 3, 5, 33])
@pytest.mark.parametrize("M", [1, 65, 300])   # one point, one past a block of single lanes, several blocks
def test_all_products(shape, J, C, M):
    from paper_2111_02912_gb300 import Plan
    case = make_case(shape, M, C, True, seed=630 + M)
    op, S = KBNufft(shape, case["omega"], J=J), case["smaps"]
    plan = Plan(shape, to_dev(case["omega"]), J=J, max_coils=C)
    x, Sd, v, dom = (to_dev(case[k]) for k in ("x", "smaps", "v", "domega"))
    y_ref = jb.sense_forward(op, case["x"], S)
    dy_ref = jb.jvp_omega(op, case["x"], case["domega"], S)
    go_ref, _ = jb.vjp_omega_x(op, case["x"], case["v"], S)
    assert rel(host(plan.forward(x, Sd)), y_ref) < TOL
    dy, y = plan.jvp_omega(x, dom, Sd, want_y=True)
    assert rel(host(dy), dy_ref) < TOL and rel(host(y), y_ref) < TOL
    assert rel(host(plan.jvp_omega(x, dom, Sd)), dy_ref) < TOL
    assert rel(host(plan.vjp_omega_x(x, v, Sd, need_x=False)[0]), go_ref) < TOL
