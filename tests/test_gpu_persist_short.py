"""The persistent Algorithm-2 step with one or two Krylov steps allowed (its first step then needs more shared
memory than any later one), against the per-phase launches: the same kernels' arithmetic apart from the order
of reductions, so both paths meet the accuracy contract or both stop short of it."""
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


@pytest.mark.parametrize("prec,tol", [("mixed", 1e-10), ("fp64", 1e-12)])
@pytest.mark.parametrize("maxit", [1, 2])
@pytest.mark.parametrize("n,nt", [(40, 16), (126, 16), (600, 8)])
def test_one_or_two_steps(pd, n, nt, maxit, prec, tol):
    P = W.heat1d_forced(n, nt, 1.0, seed=n)
    out = []
    for persistent in (1, -1):
        with pd.Plan.from_problem(P, precision=prec, alpha=1e-4, maxit=maxit, tune={"persistent": persistent}) as plan:
            U, st = plan.solve(torch.from_numpy(P.G).cuda())
            assert st["persistent_step"] == (1 if persistent == 1 else 0)
            out.append(R.rel_err(U.cpu().numpy(), R.be_solve_refined(P)))
    assert max(out) <= tol
