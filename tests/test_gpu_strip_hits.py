"""Hit lists collected per block (3-D, and 2-D from 100,000 points) and the two-stream VJP beyond 16 coils, against the oracle."""
import numpy as np
import pytest

from gpu_helpers import host, make_case, rel, to_dev
from oracle import jacobian as jb
from oracle.nufft import KBNufft

pytestmark = pytest.mark.gpu

TOL = 1e-5   # FP32 rounding of transforms, taps and hit sums: the tolerance of the parity tests


@pytest.mark.parametrize("shape,M,spread_out", [
    ((40, 34), 99999, True), ((40, 34), 100000, True), ((40, 34), 100000, False),   # either side of the rule, one place
    ((24, 20, 18), 257, True),          # one point past a block; its points far apart: many units per block
    ((64, 40, 48), 6000, True),         # more units per block than table slots
    ((20, 18, 16), 5000, False),
])
def test_hits_collected_per_block(shape, M, spread_out):
    from paper_2111_02912_gb300 import Plan
    case = make_case(shape, M, 1, False, seed=500)
    om = case["omega"] if spread_out else np.repeat(case["omega"][:, :1], M, axis=1)
    op = KBNufft(shape, om)
    for det in (False, True):
        if det and not spread_out:
            continue   # orders every point of a bin against every other
        x = Plan(shape, to_dev(om), max_coils=1, deterministic=det).adjoint(to_dev(case["y"]))
        assert rel(host(x), np.stack([op.adjoint(v) for v in case["y"]])) < TOL


@pytest.mark.parametrize("C", [17, 32, 40])
def test_two_stream_vjp_with_partial_coil_sums(C):
    """More than 16 coils: the last inverse pass sums coil chunks beside the omega-gradient chain."""
    from paper_2111_02912_gb300 import Plan
    shape, M = (40, 32), 700
    case = make_case(shape, M, C, True, seed=510)
    plan = Plan(shape, to_dev(case["omega"]), max_coils=C)
    go_ref, gx_ref = jb.vjp_omega_x(KBNufft(shape, case["omega"]), case["x"], case["v"], case["smaps"])
    for _ in range(3):   # repeated: a race between the two chains would show
        go, gx = plan.vjp_omega_x(to_dev(case["x"]), to_dev(case["v"]), to_dev(case["smaps"]))
        assert rel(host(go), go_ref) < TOL and rel(host(gx), gx_ref) < TOL
