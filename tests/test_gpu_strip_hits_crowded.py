"""The rule by which crowded 2-D strip units have their hits collected per block, on both its sides, against the oracle."""
import numpy as np
import pytest

from gpu_helpers import host, make_case, rel, to_dev
from oracle.nufft import KBNufft

pytestmark = pytest.mark.gpu

TOL = 1e-5   # FP32 rounding of transforms, taps and hit sums: the tolerance of the parity tests


@pytest.mark.parametrize("shape,C,M", [
    ((40, 34), 1, 16383), ((40, 34), 1, 16384),       # the fewest points; 15 units
    ((256, 256), 1, 16384), ((256, 256), 1, 16383),   # 512 units of 32 points each, one point fewer
    ((64, 48), 9, 20000),                             # a coil group of 16: units of four rows
])
@pytest.mark.parametrize("det", [False, True])
def test_either_side_of_the_rule(shape, C, M, det):
    from paper_2111_02912_gb300 import Plan
    case = make_case(shape, M, C, False, seed=520)
    plan = Plan(shape, to_dev(case["omega"]), max_coils=C, deterministic=det)
    x = host(plan.adjoint(to_dev(case["y"])))
    op = KBNufft(shape, case["omega"])
    assert rel(x, np.stack([op.adjoint(v) for v in case["y"]])) < TOL
