"""Line passes on either side of the rules that choose their form, against the oracle."""
import pytest

from gpu_helpers import host, make_case, rel, to_dev
from oracle import jacobian as jb
from oracle.nufft import KBNufft

pytestmark = pytest.mark.gpu

TOL = 1e-5   # FP32 rounding of transforms and taps: the tolerance of the parity tests


def _check(shape, C, maps=True, M=150):
    from paper_2111_02912_gb300 import Plan
    case = make_case(shape, M, C, maps, seed=620)
    op, S = KBNufft(shape, case["omega"]), case["smaps"]
    plan = Plan(shape, to_dev(case["omega"]), max_coils=C)
    x, Sd, v = (to_dev(case[k]) for k in ("x", "smaps", "v"))
    go_ref, gx_ref = jb.vjp_omega_x(op, case["x"], case["v"], S)
    go, gx = plan.vjp_omega_x(x, v, Sd)
    assert rel(host(plan.forward(x, Sd)), jb.sense_forward(op, case["x"], S)) < TOL
    assert rel(host(go), go_ref) < TOL and rel(host(gx), gx_ref) < TOL


@pytest.mark.parametrize("C,maps", [(1, True), (9, True), (3, False)])
@pytest.mark.parametrize("shape", [(14, 256), (256, 14), (12, 512), (12, 320), (10, 8, 256)])   # staged, and 640 not
def test_first_pass_through_shared_memory(shape, C, maps):
    _check(shape, C, maps)


@pytest.mark.parametrize("C", [1, 2])
@pytest.mark.parametrize("maps", [True, False])
@pytest.mark.parametrize("shape", [(14, 100), (14, 108), (12, 288), (8, 10, 108), (108,), (216,)])   # 200 points, 216, 576
def test_last_pass_of_a_single_channel(shape, C, maps):
    _check(shape, C, maps)


@pytest.mark.parametrize("C", [1, 8, 17])
@pytest.mark.parametrize("shape", [(160, 14), (14, 10, 72), (72, 14, 10), (10, 72, 14)])   # 8 lines, 16 on each 3-D axis
def test_middle_pass_heights(shape, C):
    _check(shape, C)
