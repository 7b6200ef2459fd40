"""JVP with values of eight coils, whole lines and (odd taps, 2-D) coil pairs, against the oracle."""
import pytest

from gpu_helpers import host, make_case, rel, to_dev
from oracle import jacobian as jb
from oracle.nufft import KBNufft

pytestmark = pytest.mark.gpu

TOL = 1e-5   # FP32 rounding of transforms and taps: the tolerance of the parity tests


@pytest.mark.parametrize("shape", [(24, 20), (26, 22), (12, 14, 12)])
@pytest.mark.parametrize("J", [4, 5, 6, 7, 8])
@pytest.mark.parametrize("M", [17, 700])
def test_values_and_derivative(shape, J, M):
    from paper_2111_02912_gb300 import Plan
    case = make_case(shape, M, 8, True, seed=640 + M)
    op, S = KBNufft(shape, case["omega"], J=J), case["smaps"]
    plan = Plan(shape, to_dev(case["omega"]), J=J, max_coils=8)
    dy, y = plan.jvp_omega(to_dev(case["x"]), to_dev(case["domega"]), to_dev(S), want_y=True)
    assert rel(host(y), jb.sense_forward(op, case["x"], S)) < TOL
    assert rel(host(dy), jb.jvp_omega(op, case["x"], case["domega"], S)) < TOL
