"""The one-launch sort of small strip plans: edges of its range against the oracle, and its hand-over to the separate launches."""
import numpy as np
import pytest

from gpu_helpers import host, make_case, rel, to_dev
from oracle.nufft import KBNufft

pytestmark = pytest.mark.gpu

TOL = 1e-5   # FP32 rounding of transforms, taps and hit sums: the tolerance of the parity tests


def _check(plan, shape, om, y, x):
    op = KBNufft(shape, om)
    assert rel(host(plan.adjoint(to_dev(y))), np.stack([op.adjoint(v) for v in y])) < TOL
    assert rel(host(plan.forward(to_dev(x))), np.stack([op.forward(v) for v in x])) < TOL


@pytest.mark.parametrize("shape,M", [
    ((40, 34), 1), ((40, 34), 31), ((40, 34), 33),            # less than a warp, one past it
    ((40, 34), 4097), ((40, 34), 32768), ((40, 34), 32769),   # one past the cluster's threads, the last size, the next
    ((20, 18, 16), 5), ((20, 18, 16), 4100),
    ((300, 280), 900),                                        # more bins and units than threads of a block
])
def test_small_sort_matches_the_oracle(shape, M):
    from paper_2111_02912_gb300 import Plan
    case = make_case(shape, M, 2, False, seed=400)
    _check(Plan(shape, to_dev(case["omega"]), max_coils=2), shape, case["omega"], case["y"], case["x"])


@pytest.mark.parametrize("M", [64, 65, 4097, 20000])
def test_points_in_one_place_are_split(M):
    """Every hit in the same few units: parts, their length doubled where the slots run out."""
    from paper_2111_02912_gb300 import Plan
    shape = (40, 34)
    case = make_case(shape, M, 1, False, seed=401)
    om = np.repeat(np.array([[0.3], [-0.7]], np.float32), M, axis=1)
    _check(Plan(shape, to_dev(om), max_coils=1), shape, om, case["y"], case["x"])


def test_small_and_large_point_sets_in_turn_and_in_a_graph():
    import torch

    from paper_2111_02912_gb300 import Plan
    shape = (40, 34)
    cases = [make_case(shape, M, 2, False, seed=410 + k) for k, M in enumerate((700, 40000, 900, 32768))]
    plan = Plan(shape, to_dev(cases[1]["omega"]), max_coils=2)
    for c in cases + cases[:2]:
        plan.set_points(to_dev(c["omega"]))
        _check(plan, shape, c["omega"], c["y"], c["x"])
    om, y = to_dev(cases[0]["omega"]), to_dev(cases[0]["y"])
    plan.set_points(om)
    plan.adjoint(y)
    torch.cuda.synchronize()
    g, out = torch.cuda.CUDAGraph(), torch.empty((2,) + shape, dtype=torch.complex64, device="cuda")
    with torch.cuda.graph(g):
        plan.set_points(om)
        plan.adjoint(y, out=out)
    other = make_case(shape, 700, 2, False, seed=420)
    om.copy_(to_dev(other["omega"]))
    for _ in range(2):   # every replay sorts anew
        g.replay()
        torch.cuda.synchronize()
        op = KBNufft(shape, other["omega"])
        assert rel(host(out), np.stack([op.adjoint(v) for v in cases[0]["y"]])) < TOL
