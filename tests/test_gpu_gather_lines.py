"""The eight-coil whole-line gathers against the oracle, and against the pair gathers where it has no counterpart."""
import numpy as np
import pytest

from gpu_helpers import host, make_case, rel, to_dev
from oracle import jacobian as jb
from oracle.nufft import KBNufft

pytestmark = pytest.mark.gpu

# FP32 rounding of the transforms and of J^D <= 512 accumulated taps: the tolerance of the parity tests.
TOL = 1e-5


@pytest.mark.parametrize("shape,J,sigma", [
    ((24, 20), 6, 2.0), ((24, 30), 4, 2.0), ((20, 24), 5, 1.25), ((26, 22), 7, 2.0), ((24, 20), 8, 2.0),
    ((14, 16, 12), 6, 2.0), ((16, 12, 14), 5, 1.25), ((12, 12, 16), 8, 2.0), ((12, 16, 12), 4, 2.0), ((12, 14, 12), 7, 2.0),
])
@pytest.mark.parametrize("M", [1, 17, 700])   # one point, one point past a block, many
def test_eight_coil_gathers(shape, J, sigma, M):
    from paper_2111_02912_gb300 import Plan
    case = make_case(shape, M, 8, True, seed=300 + M)
    om = case["omega"]
    op = KBNufft(shape, om, J=J, sigma=sigma)
    if M > 4:   # windows around the end of the last axis, starting at even and odd columns, a third of a cell in
        om[-1, :4] = (2 * np.pi / op.K[-1]) * (np.array([-1.0, 0.0, 1.0, 2.0]) + 1 / 3)
        op = KBNufft(shape, om, J=J, sigma=sigma)
    x, S, v, dom = (to_dev(case[k]) for k in ("x", "smaps", "v", "domega"))
    lines = Plan(shape, to_dev(om), J=J, sigma=sigma, max_coils=8)
    pairs = Plan(shape, to_dev(om), J=J, sigma=sigma, max_coils=8, gather="pairs")
    y = lines.forward(x, S)
    assert rel(host(y), jb.sense_forward(op, case["x"], case["smaps"])) < TOL
    go_ref, gx_ref = jb.vjp_omega_x(op, case["x"], case["v"], case["smaps"])
    go, gx = lines.vjp_omega_x(x, v, S)
    assert rel(host(go), go_ref) < TOL and rel(host(gx), gx_ref) < TOL
    for want_y in (False, True):
        got, want = lines.jvp_omega(x, dom, S, want_y=want_y), pairs.jvp_omega(x, dom, S, want_y=want_y)
        for a, b in zip(got if want_y else (got,), want if want_y else (want,)):
            assert rel(host(a), host(b)) < TOL
