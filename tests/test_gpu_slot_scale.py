"""The batches' exact per-problem scaling inside the transforms: problems of very different magnitude,
unused slots, both dimensions, every length class of the time DFT and of the DST, and a graph that
serves several right-hand sides in turn.  Bound: each problem against the oracle, relative to its own
norm, the accuracy contract of the path."""
import numpy as np
import pytest

import workloads as W
from oracle import reference as R

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {"mixed": 1e-10, "fp64": 1e-12}


@pytest.fixture(scope="module")
def pd():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as entry

    entry.build()
    import paper_2304_12597_gb300 as pkg

    return pkg


def _check(plan, probs, mags, prec, U):
    Uh = U.cpu().numpy()
    for P, A, m in zip(probs, plan.unstack(Uh, [P.nx * P.ny for P in probs], [P.nt for P in probs]), mags):
        if m == 0.0:
            assert not A.any()
        else:
            assert R.rel_err(A, m * R.be_solve_refined(P)) < TOL[prec], m
    # columns that hold no unknown come back as exact zeros
    V = Uh.reshape(plan.nt, plan.batch, plan.slot)
    for b, P in enumerate(probs):
        assert not V[:, b, P.nx * P.ny:].any()


MAGS = (1.0, 1e-120, 0.0, 3e130, 7e-9)


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("dim,nt", [(1, 8), (1, 64), (1, 512), (1, 2048), (1, 4096), (2, 16), (2, 256)])
def test_magnitudes_and_unused_slots(pd, dim, nt, prec):
    if dim == 1:
        probs = [W.heat1d_forced(n, nt, 1.0, seed=n) for n in (33, 20, 17, 40, 9)]
    else:
        n = 63 if nt == 256 else 15  # (the half-extension transform and the general one)
        probs = [W.heat2d_smooth(n, nt, 0.1, seed=s) for s in range(5)]
    rng = np.random.default_rng(0)
    with pd.Plan.from_problems(probs, precision=prec, alpha=1e-2) as plan:
        U = torch.full((plan.nt, plan.nbar), float("nan"), dtype=torch.float64, device="cuda")
        for mags in (MAGS, tuple(rng.permutation(MAGS))):  # one captured graph, other buffers and scales
            G = torch.from_numpy(plan.stack([m * P.G for P, m in zip(probs, mags)])).cuda()
            plan.solve(G, U)
            _check(plan, probs, mags, prec, U)
        # the same through sweep-by-sweep advances
        U.fill_(float("nan"))
        state, _ = plan.advance(G, U, [1] * plan.batch, steps=1)
        for _ in range(20):
            if all(s == 1 or m == 0.0 for s, m in zip(state, mags)):
                break
            state, _ = plan.advance(G, U, [0] * plan.batch, steps=1)
        _check(plan, probs, mags, prec, U)
