"""Deterministic plans: the bits depend on the points, not on how many the plan has held before."""
import numpy as np
import pytest

from gpu_helpers import make_case, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,C,before", [((256, 256), 4, 65537), ((40, 48, 44), 2, 60000)])   # over 256 units
def test_fresh_and_used_plans_agree_bitwise(shape, C, before):
    """Points near the k-space centre, whose units are split: into the same parts by a fresh plan and by
    one whose storage has grown for many more points."""
    import torch

    from paper_2111_02912_gb300 import Plan
    M = 6000
    case = make_case(shape, M, C, False, seed=900)
    g = np.random.default_rng(901)
    om = to_dev(np.clip(g.normal(0.0, 0.1, (len(shape), M)), -np.pi, np.pi).astype(np.float32))
    many = to_dev(np.clip(g.normal(0.0, 1.0, (len(shape), before)), -np.pi, np.pi).astype(np.float32))
    y, x = to_dev(case["y"]), to_dev(case["x"])
    fresh = Plan(shape, om, max_coils=C, deterministic=True)
    used = Plan(shape, many, max_coils=C, deterministic=True)
    used.set_points(om)
    assert torch.equal(torch.view_as_real(fresh.adjoint(y)), torch.view_as_real(used.adjoint(y)))
    for a, b in zip(fresh.vjp_omega_x(x, y), used.vjp_omega_x(x, y)):
        assert torch.equal(torch.view_as_real(a) if a.is_complex() else a, torch.view_as_real(b) if b.is_complex() else b)
