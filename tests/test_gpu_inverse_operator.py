"""psd_inverse solves with the operator that it is given: replaced methods, of the object, its class or its
plan, are what the iteration applies, and b's values count, not its storage."""
import pytest

from gpu_helpers import host, make_case, rel, to_dev
from test_gpu_cg import TOL

pytestmark = pytest.mark.gpu

SHAPE, M, C, LAM, ITERS = (24, 20), 700, 3, 350.0, 4


def _operator(seed):
    from paper_2111_02912_gb300.autograd import NufftOperator
    case = make_case(SHAPE, M, C, True, seed=seed)
    om = to_dev(case["omega"])
    return om, to_dev(case["x"]), NufftOperator(SHAPE, om, smaps=to_dev(case["smaps"]))


@pytest.mark.parametrize("where", ["class", "plan class", "plan", "another operator's"])
def test_replaced_methods_are_applied(where, monkeypatch):
    from paper_2111_02912_gb300 import Plan
    from paper_2111_02912_gb300.autograd import NufftOperator, cg_solve, psd_inverse
    om, b, op = _operator(94)
    if where == "another operator's":
        _, _, other = _operator(95)
        op.forward, op.adjoint = other.forward, other.adjoint
    else:
        target = {"class": NufftOperator, "plan class": Plan, "plan": op.plan}[where]
        for name in ("forward", "adjoint"):
            plain = getattr(target, name)
            monkeypatch.setattr(target, name, lambda *a, plain=plain, **k: 2.0 * plain(*a, **k))
    want = cg_solve(lambda v: op.adjoint(op.forward(v)) + LAM * v, b, ITERS)
    assert rel(host(psd_inverse(b, om, op, LAM, ITERS)), host(want)) < TOL


def test_values_of_a_negative_view():
    import torch

    from paper_2111_02912_gb300.autograd import psd_inverse
    om, b, op = _operator(96)
    got, want = psd_inverse(torch._neg_view(b), om, op, LAM, ITERS), psd_inverse(b, om, op, LAM, ITERS)
    assert rel(host(got), -host(want)) < TOL
