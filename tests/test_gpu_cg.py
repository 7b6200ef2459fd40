"""The library's CG on (E'E + lam I) x = b against the same iteration on the oracle's operator in FP64."""
import numpy as np
import pytest

from gpu_helpers import host, make_case, rel, to_dev
from oracle import jacobian as jb
from oracle.nufft import KBNufft

pytestmark = pytest.mark.gpu

# Four iterations from zero with lam of the size of the spectrum: the iterates are polynomials of
# degree four of a matrix of condition number below about 10, so the 2e-7 of one FP32 normal product
# grows by less than the sum of its coefficients, some tens: 1e-5.
TOL = 1e-5


def _cg(F, b, iters):
    x, r = np.zeros_like(b), b.copy()
    p, rr = r.copy(), np.vdot(b, b).real
    for _ in range(iters):
        q = F(p)
        al = rr / np.vdot(p, q).real
        x, r = x + al * p, r - al * q
        rn = np.vdot(r, r).real
        p, rr = r + (rn / rr) * p, rn
    return x


@pytest.mark.parametrize("shape,M,C,maps,spread", [
    ((10, 12), 150, 3, True, "general"),      # fewer elements than one block
    ((24, 20), 700, 5, True, "auto"),         # strips, an odd coil count
    ((40, 34), 900, 17, True, "auto"),        # two coil groups in the sorted k-space values
    ((24, 20), 700, 4, False, "auto"),        # one system over several images
    ((64,), 300, 2, True, "auto"),            # 1-D: k-space values in the work buffer
    ((16, 14, 12), 900, 3, True, "auto"),     # 3-D strips
    ((512, 400), 3000, 1, True, "auto"),      # more elements than blocks times threads
    ((24, 20), 0, 2, True, "auto"),           # no points: x = b / lam after one step
])
def test_cg_matches_the_oracle(shape, M, C, maps, spread):
    from paper_2111_02912_gb300 import Plan
    iters, lam = 4, 0.5 * max(M, 1)
    case = make_case(shape, max(M, 1), C, maps, seed=91)
    om, S = case["omega"][:, :M], case["smaps"]
    b = case["x"]
    plan = Plan(shape, to_dev(np.ascontiguousarray(om)), max_coils=C, spread=spread)
    x = host(plan.cg_normal(to_dev(b), lam, 1 if M == 0 else iters, to_dev(S) if maps else None))
    if M == 0:
        assert rel(x, b / lam) < TOL
        return
    op = KBNufft(shape, om)
    if maps:
        F = lambda v: jb.sense_adjoint(op, jb.sense_forward(op, v, S), S) + lam * v
    else:
        F = lambda v: np.stack([op.adjoint(op.forward(w)) for w in v]) + lam * v
    assert rel(x, _cg(F, b.astype(np.complex128), iters)) < TOL


def test_inverse_of_a_conjugate_view_and_of_a_replaced_operator():
    """psd_inverse takes the library's solver for a plain operator only, and reads b's values, not its storage."""
    import torch

    from paper_2111_02912_gb300.autograd import NufftOperator, cg_solve, psd_inverse
    case = make_case((24, 20), 700, 3, True, seed=92)
    om, b = to_dev(case["omega"]), to_dev(case["x"])
    op = NufftOperator((24, 20), om, smaps=to_dev(case["smaps"]))
    F = lambda v: op.adjoint(op.forward(v)) + 350.0 * v
    got = psd_inverse(b.conj(), om, op, 350.0, 4)
    assert rel(host(got), host(cg_solve(F, b.conj().resolve_conj(), 4))) < TOL
    calls = []
    plain = op.forward
    op.forward = lambda x: (calls.append(1), 2.0 * plain(x))[1]
    op.adjoint = lambda y, E=op.adjoint: 2.0 * E(y)
    got = psd_inverse(b, om, op, 350.0, 4)
    assert len(calls) == 4
    assert rel(host(got), host(cg_solve(F, b, 4))) < TOL
    assert torch.isfinite(torch.view_as_real(got)).all()
