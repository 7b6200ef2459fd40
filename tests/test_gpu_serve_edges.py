"""A reconstruction request with an iteration count that is not positive returns zeros."""
import pytest

from gpu_helpers import host, make_case, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("iters", [0, -1])
def test_no_iterations(iters):
    from paper_2111_02912_gb300.serve import Request, Server
    case = make_case((24, 20), 300, 2, True, seed=62)
    srv = Server(budget_bytes=1 << 30, slots=1)
    srv.submit(Request(0, "recon", case["shape"], to_dev(case["omega"]), to_dev(case["smaps"]), y=to_dev(case["y"]),
                       lam=1.0, iters=iters))
    done = srv.drain()
    assert len(done) == 1 and done[0].result.shape == case["shape"] and not host(done[0].result).any()
