"""Solves of the longest time axes: 4096 steps in binary64 and 8192 in both precisions (the z sum's
weights then take 32 KB and more of shared memory)."""
import pytest

import workloads as W
from oracle import reference as R

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("mixed", 1e-10)])
@pytest.mark.parametrize("nt", [4096, 8192])
def test_long_time_axis(prec, tol, nt):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as entry

    entry.build()
    from paper_2304_12597_gb300 import Plan

    P = W.heat1d_forced(21, nt, 1.0, seed=1)
    with Plan.from_problem(P, precision=prec) as plan:
        U, _ = plan.solve(torch.from_numpy(P.G).cuda())
    assert R.rel_err(U.cpu().numpy(), R.be_solve_refined(P)) < tol
