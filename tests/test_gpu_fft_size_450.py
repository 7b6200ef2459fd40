"""Grid edge 450 at sigma = 2, which the image sides 218 to 224 have, on either axis, against the oracle."""
import pytest

from gpu_helpers import host, make_case, rel, to_dev
from oracle import jacobian as jb
from oracle.nufft import KBNufft

pytestmark = pytest.mark.gpu

TOL = 1e-5   # FP32 rounding of transforms and taps: the tolerance of the parity tests


@pytest.mark.parametrize("last", [True, False])
@pytest.mark.parametrize("n,C", [(218, 1), (218, 9), (224, 5), (224, 17)])
def test_line_length_450(n, C, last):
    from paper_2111_02912_gb300 import Plan
    shape = (22, n) if last else (n, 22)
    case = make_case(shape, 200, C, True, seed=601)
    op = KBNufft(shape, case["omega"])
    assert 450 in op.K
    plan = Plan(shape, to_dev(case["omega"]), max_coils=C)
    x, S, v = (to_dev(case[k]) for k in ("x", "smaps", "v"))
    go_ref, gx_ref = jb.vjp_omega_x(op, case["x"], case["v"], case["smaps"])
    go, gx = plan.vjp_omega_x(x, v, S)
    assert rel(host(plan.forward(x, S)), jb.sense_forward(op, case["x"], case["smaps"])) < TOL
    assert rel(host(go), go_ref) < TOL and rel(host(gx), gx_ref) < TOL
