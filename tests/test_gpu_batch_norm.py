"""The batches' scale exponents from binary32 squares (csrc/batch.cu): slot widths around the lanes of a
row and the loads in flight, magnitudes up to the ends of what binary64 squares hold, and infinities.
Bound: each problem against the oracle, relative to its own norm, the accuracy contract of the path."""
import numpy as np
import pytest

import workloads as W
from oracle import reference as R

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pd():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as entry

    entry.build()
    import paper_2304_12597_gb300 as pkg

    return pkg


@pytest.mark.parametrize("n,nt", [(1, 64), (31, 16), (33, 256), (255, 64), (257, 8), (1500, 32)])
def test_widths_and_magnitudes(pd, n, nt):
    probs = [W.heat1d_forced(n, nt, 1.0, seed=s) for s in range(6)]
    mags = (1e-152, 1.0, 0.0, 1e-300, 1e148, 3e-150)
    with pd.Plan.from_problems(probs, precision="mixed", alpha=1e-2) as plan:
        G = torch.from_numpy(plan.stack([m * P.G for P, m in zip(probs, mags)])).cuda()
        U, _ = plan.solve(G)
        for P, A, m in zip(probs, plan.unstack(U.cpu().numpy(), [n] * 6), mags):
            if m in (0.0, 1e-300):  # its squares are zero: an unused slot
                assert not A.any()
            else:
                assert R.rel_err(A / m, R.be_solve_refined(P)) < 1e-10, m


@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
def test_a_non_finite_problem_is_reported(pd, bad):
    probs = [W.heat1d_forced(63, 64, 1.0, seed=s) for s in range(3)]
    with pd.Plan.from_problems(probs, precision="mixed") as plan:
        G = plan.stack([P.G for P in probs])
        G[5, 70] = bad
        with pytest.raises(pd.ParadiagError) as e:
            plan.solve(torch.from_numpy(G).cuda())
        assert e.value.status_name == "PD_ERR_NONFINITE"
