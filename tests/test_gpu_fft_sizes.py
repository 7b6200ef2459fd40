"""Line lengths of the second two-phase list, on either axis, with and without compile-time pruning, against the oracle."""
import pytest

from gpu_helpers import host, make_case, rel, to_dev
from oracle import jacobian as jb
from oracle.nufft import KBNufft

pytestmark = pytest.mark.gpu

TOL = 1e-5   # FP32 rounding of transforms and taps: the tolerance of the parity tests
LENGTHS = (120, 144, 180, 200, 216, 288, 300, 360, 432, 450, 576)


@pytest.mark.parametrize("last", [True, False])        # first and last pass, or the middle passes
@pytest.mark.parametrize("C", [1, 9])                  # part of a tile of lines; two coil chunks
@pytest.mark.parametrize("sigma", [2.0, 1.25])
@pytest.mark.parametrize("L", LENGTHS)
def test_line_length(L, sigma, C, last):
    from paper_2111_02912_gb300 import Plan
    n = L // 2 if sigma == 2.0 else 2 * int(L / sigma / 2)   # sigma n just below L, which is then the grid edge
    shape = (22, n) if last else (n, 22)
    if n % 2:
        pytest.skip("image sides are even")
    case = make_case(shape, 200, C, True, seed=600)
    op = KBNufft(shape, case["omega"], sigma=sigma)
    if L not in op.K:
        pytest.skip("no image side has this grid edge at this sigma")
    plan = Plan(shape, to_dev(case["omega"]), sigma=sigma, max_coils=C)
    x, S, v = (to_dev(case[k]) for k in ("x", "smaps", "v"))
    go_ref, gx_ref = jb.vjp_omega_x(op, case["x"], case["v"], case["smaps"])
    go, gx = plan.vjp_omega_x(x, v, S)
    assert rel(host(plan.forward(x, S)), jb.sense_forward(op, case["x"], case["smaps"])) < TOL
    assert rel(host(go), go_ref) < TOL and rel(host(gx), gx_ref) < TOL


@pytest.mark.parametrize("n", [20, 72, 90, 250, 320])   # 1-D, one channel: a tile of a single line
def test_single_line(n):
    from paper_2111_02912_gb300 import Plan
    case = make_case((n,), 60, 1, True, seed=610)
    op = KBNufft((n,), case["omega"])
    plan = Plan((n,), to_dev(case["omega"]), max_coils=1)
    x, S, v = (to_dev(case[k]) for k in ("x", "smaps", "v"))
    go_ref, gx_ref = jb.vjp_omega_x(op, case["x"], case["v"], case["smaps"])
    go, gx = plan.vjp_omega_x(x, v, S)
    assert rel(host(plan.forward(x, S)), jb.sense_forward(op, case["x"], case["smaps"])) < TOL
    assert rel(host(go), go_ref) < TOL and rel(host(gx), gx_ref) < TOL
