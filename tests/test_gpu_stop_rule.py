"""Refinement of near-singular problems in mixed precision (heat with almost insulated ends): the sweeps'
Algorithm 2 stops at very different residuals, so the ratio of the last two updates alone says little about
what the last sweep left.  Every solution meets the accuracy contract of the mixed path, 1e-10 relative
2-norm against the oracle."""
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


def _insulated(n, nt, T, seed):
    P = W.heat1d_forced(n, nt, T, seed=seed)
    P.k_diag[0] += 0.999 * P.k_up[0]
    P.k_diag[-1] += 0.999 * P.k_lo[-1]
    return P


@pytest.mark.parametrize("n,nt,T,seed", [(248, 64, 1.3787817640067888, 152648422), (79, 128, 3.2890412811822745, 801299469),
                                         (200, 128, 1.3141721875863261, 162589093), (92, 8, 2.4997650143321515, 61807406),
                                         (85, 32, 2.963323483834398, 347893066), (313, 16, 1.5429647755198193, 663796830),
                                         (112, 8, 3.221330443986384, 761827613)])
def test_single_problems(pd, n, nt, T, seed):
    P = _insulated(n, nt, T, seed)
    with pd.Plan.from_problem(P, precision="mixed") as plan:
        U, st = plan.solve(torch.from_numpy(P.G).cuda())
    assert R.rel_err(U.cpu().numpy(), R.be_solve_refined(P)) <= 1e-10, st


@pytest.mark.parametrize("scale", [2.0 ** -46, 2.0 ** -50])
@pytest.mark.parametrize("n,nt,T,seed", [(200, 128, 1.3141721875863261, 162589093), (92, 8, 2.4997650143321515, 61807406),
                                         (6, 4, 0.05245022822372974, 445)])
def test_updates_below_the_range_of_binary32_squares(pd, n, nt, T, seed, scale):
    """Right-hand sides so small that the squares of a sweep's update underflow in binary32."""
    P = _insulated(n, nt, T, seed)
    with pd.Plan.from_problem(P, precision="mixed") as plan:
        U, st = plan.solve(torch.from_numpy(P.G * scale).cuda())
    assert R.rel_err(U.cpu().numpy() / scale, R.be_solve_refined(P)) <= 1e-10, st


@pytest.mark.parametrize("n,nt", [(3, 64), (117, 64), (200, 128), (79, 128)])
@pytest.mark.parametrize("advance", [False, True])
def test_batches(pd, n, nt, advance):
    probs = [_insulated(n, nt, T, seed) for T, seed in ((1.6, 995733192), (0.1, 7), (1.3, 162589093), (3.3, 801299469))]
    probs += [W.heat1d_forced(n, nt, 1.0, seed=1), W.advdiff1d_pulse(n, nt, seed=2)]
    with pd.Plan.from_problems(probs, precision="mixed") as plan:
        G = torch.from_numpy(plan.stack([P.G for P in probs])).cuda()
        if advance:
            U = torch.empty_like(G)
            state, _ = plan.advance(G, U, [1] * len(probs))
            while 0 in state:
                state, st = plan.advance(G, U, [0] * len(probs))
            assert state == [1] * len(probs)
        else:
            U, st = plan.solve(G)
        parts = plan.unstack(U.cpu().numpy(), [n] * len(probs))
    for P, A in zip(probs, parts):
        assert R.rel_err(A, R.be_solve_refined(P)) <= 1e-10, st
