"""Which operators psd_inverse hands to the library's solver: those that call their own methods (no GPU)."""
import pytest

from paper_2111_02912_gb300 import autograd as ag


def _operator():
    op = object.__new__(ag.NufftOperator)
    op.plan = object.__new__(ag.Plan)
    op.plan.handle = None
    return op


class _Sub(ag.NufftOperator):
    pass


def test_plain_operators_only():
    op = _operator()
    assert ag._applies_own_methods(op)
    assert not ag._applies_own_methods(object())
    sub = object.__new__(_Sub)
    sub.plan = op.plan
    assert not ag._applies_own_methods(sub)
    op.forward = _operator().forward                       # bound to another operator
    assert not ag._applies_own_methods(op)


@pytest.mark.parametrize("name", ["forward", "adjoint"])
@pytest.mark.parametrize("where", ["class", "plan class", "operator", "plan"])
def test_a_replaced_method_is_noticed(where, name, monkeypatch):
    op = _operator()
    target = {"class": ag.NufftOperator, "plan class": ag.Plan, "operator": op, "plan": op.plan}[where]
    monkeypatch.setattr(target, name, lambda *a, **k: None)
    assert not ag._applies_own_methods(op)
