"""Default part lengths of split strip units, from the shortest to those that the heaviest unit calls for,
against the oracle."""
import numpy as np
import pytest

from gpu_helpers import host, make_case, rel, to_dev
from oracle.nufft import KBNufft

pytestmark = pytest.mark.gpu

TOL = 1e-5   # FP32 rounding of transforms, taps and hit sums: the tolerance of the parity tests


# hits of the heaviest unit: 32 to a part up to 341, 64 up to 1365, then 128 and 256 (and longer for the slots)
@pytest.mark.parametrize("heavy", [341, 342, 1366, 5462, 30000])
@pytest.mark.parametrize("shape", [(40, 34), (20, 18, 16)])
@pytest.mark.parametrize("det", [False, True])
def test_one_heavy_unit_among_light_ones(heavy, shape, det):
    from paper_2111_02912_gb300 import Plan
    if det and heavy > 6000:
        pytest.skip("orders every point of a bin against every other")
    M = heavy + 400
    case = make_case(shape, M, 1, False, seed=530)
    om = case["omega"].copy()
    om[:, :heavy] = np.linspace(0.3, 0.9, len(shape), dtype=np.float32)[:, None]
    plan = Plan(shape, to_dev(om), max_coils=1, deterministic=det)
    x = host(plan.adjoint(to_dev(case["y"])))
    op = KBNufft(shape, om)
    assert rel(x, np.stack([op.adjoint(v) for v in case["y"]])) < TOL


# units of even weight: many of them (whole), few (cut); and hardly any hits to a unit
@pytest.mark.parametrize("shape,M,C", [((256, 256), 30000, 8), ((40, 34), 30000, 1), ((40, 34), 700, 2), ((36, 40, 44), 20000, 2)])
def test_units_of_even_weight(shape, M, C):
    from paper_2111_02912_gb300 import Plan
    case = make_case(shape, M, C, False, seed=531)
    x = host(Plan(shape, to_dev(case["omega"]), max_coils=C).adjoint(to_dev(case["y"])))
    op = KBNufft(shape, case["omega"])
    assert rel(x, np.stack([op.adjoint(v) for v in case["y"]])) < TOL
