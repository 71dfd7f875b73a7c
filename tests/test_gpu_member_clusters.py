"""The vector steps of a batch's Algorithm 2 on a thread-block cluster per problem against one CTA per
problem (krylov_cluster = -1), for every cluster size the rule picks and numbers of entries per thread,
ragged problems, unused slots, and problems that stop at different steps.

Both paths meet the bars (1e-10 mixed, 1e-12 FP64), so they agree within twice that (relative 2-norm,
each problem by itself)."""
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


@pytest.mark.parametrize("prec,tol", [("mixed", 2e-10), ("fp64", 2e-12)])
# clusters of 8 and 4, 38 problems the last that fit, none (too many problems), none (short problems); 256 is
# the first length
@pytest.mark.parametrize("n,nt,batch", [(2048, 32, 8), (4096, 16, 3), (257, 64, 9), (1023, 32, 18), (1500, 16, 38),
                                        (300, 16, 40), (255, 16, 4), (256, 16, 2)])
def test_clusters_agree_with_one_cta(pd, n, nt, batch, prec, tol):
    make = [W.heat1d_forced, W.advdiff1d_pulse, W.random_tridiag_problem]
    probs = [make[i % 3](n - (i * 7) % 50, nt, seed=i) for i in range(batch)]
    out = []
    for tune in (None, {"krylov_cluster": -1}):
        with pd.Plan.from_problems(probs, precision=prec, tune=tune) as plan:
            G = plan.stack([P.G * (0.0 if i == 1 else 1.0) for i, P in enumerate(probs)])
            U, _ = plan.solve(torch.from_numpy(G).cuda())
            out.append(plan.unstack(U.cpu().numpy(), [P.nx for P in probs]))
    for i, (a, b) in enumerate(zip(*out)):
        if i == 1:
            assert not a.any() and not b.any()
        else:
            assert R.rel_err(a, b) < tol, i
    assert R.rel_err(out[0][0], R.be_solve_refined(probs[0])) < tol
