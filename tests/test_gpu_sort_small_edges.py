"""The one-launch sort (up to 4096 points, small 2-D tables, not recorded) at the edge of its range and with
parts that do not fit the partial-sum slots at first, against the oracle."""
import numpy as np
import pytest

from gpu_helpers import host, make_case, rel, to_dev
from oracle.nufft import KBNufft
from test_gpu_sort_small import TOL, _check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(40, 34), (20, 18, 16)])
@pytest.mark.parametrize("M", [4095, 4096, 4097])   # the last sizes of one launch, the first of several
def test_either_side_of_the_rule(shape, M):
    from paper_2111_02912_gb300 import Plan
    case = make_case(shape, M, 2, False, seed=800)
    _check(Plan(shape, to_dev(case["omega"]), max_coils=2), shape, case["omega"], case["y"], case["x"])


@pytest.mark.parametrize("shape,coils", [
    ((256, 256), 2),     # 1024 bins, the last size of one launch
    ((192, 192), 8),     # 1152 strip units, past one per thread
    ((256, 272), 2),     # more bins: several launches
    ((256, 256), 8),     # more units
])
@pytest.mark.parametrize("M", [900, 4096])
def test_table_sizes(shape, coils, M):
    from paper_2111_02912_gb300 import Plan
    case = make_case(shape, M, 2, False, seed=802)
    _check(Plan(shape, to_dev(case["omega"]), max_coils=coils), shape, case["omega"], case["y"], case["x"])


@pytest.mark.parametrize("M", [1000, 4096])
@pytest.mark.parametrize("part", [0, 8, 32])
@pytest.mark.parametrize("where", ["one place", "two places", "spread out"])
def test_parts_are_lengthened_until_they_fit(M, part, where):
    """One place: M hits in each of a few units, M / 8 parts each for 256 slots, so the length doubles."""
    from paper_2111_02912_gb300 import Plan
    shape = (40, 34)
    case = make_case(shape, M, 1, False, seed=801)
    om = case["omega"].copy()
    if where != "spread out":
        om[:, :] = np.array([[0.3], [-0.7]], np.float32)
    if where == "two places":
        om[:, M // 3:] = np.array([[-2.0], [3.1]], np.float32)
    _check(Plan(shape, to_dev(om), max_coils=1, strip_part=part), shape, om, case["y"], case["x"])


def test_one_launch_and_several_in_turn():
    from paper_2111_02912_gb300 import Plan
    shape = (40, 34)
    cases = [make_case(shape, M, 2, False, seed=810 + k) for k, M in enumerate((4096, 4097, 4095, 5000, 4096))]
    plan = Plan(shape, to_dev(cases[1]["omega"]), max_coils=2, strip_part=8)
    for c in cases:
        plan.set_points(to_dev(c["omega"]))
        _check(plan, shape, c["omega"], c["y"], c["x"])


def test_recorded_sorts_take_several_launches():
    """Eager and recorded sorts of one plan in turn, each from the counts that the other has left."""
    import torch

    from paper_2111_02912_gb300 import Plan
    from paper_2111_02912_gb300 import _abi
    shape, M = (40, 34), 4000
    cases = [make_case(shape, M, 2, False, seed=820 + k) for k in range(3)]
    om, y = to_dev(cases[0]["omega"]), to_dev(cases[0]["y"])
    plan = Plan(shape, om, max_coils=2)
    out = plan.adjoint(y)
    n = _abi.nufft_launch_count()
    plan.set_points(om)
    plan.sort_points()
    assert _abi.nufft_launch_count() - n == 1
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        n = _abi.nufft_launch_count()
        plan.set_points(om)
        plan.sort_points()
        assert _abi.nufft_launch_count() - n > 1
        plan.adjoint(y, out=out)
    for c in cases:
        om.copy_(to_dev(c["omega"]))
        g.replay()
        torch.cuda.synchronize()
        op = KBNufft(shape, c["omega"])
        assert rel(host(out), np.stack([op.adjoint(v) for v in cases[0]["y"]])) < TOL
        plan.set_points(to_dev(c["omega"]))
        _check(plan, shape, c["omega"], c["y"], c["x"])
