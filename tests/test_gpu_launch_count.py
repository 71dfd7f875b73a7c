"""stats.kernel_launches of solves and advance calls that run as one graph, over more sweeps than the
per-sweep tables of the statistics hold (16): the same kernels as the host-driven loops launch, so the
same count, whole numbers."""
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

KW = dict(maxit=2, max_refine=60)  # two Krylov steps a solve: slow contraction, many sweeps


@pytest.fixture(scope="module")
def pd():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as entry

    entry.build()
    import paper_2304_12597_gb300 as pkg

    return pkg


def _problem(seed):
    P = W.heat1d_forced(100, 32, 0.1, seed=seed)
    for a in (P.k_lo, P.k_diag, P.k_up):
        a *= 1e-2
    return P


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
def test_advance(pd, prec):
    probs = [_problem(0), _problem(1)]

    def run(no_graph):
        out = []
        with pd.Plan.from_problems(probs, precision=prec, no_graph=no_graph, **KW) as plan:
            G = torch.from_numpy(plan.stack([P.G for P in probs])).cuda()
            U = torch.zeros_like(G)
            for _ in range(9):
                _, st = plan.advance(G, U, [1, 1], steps=40)
                out.append((st["refine_sweeps"], st["krylov_iters_total"], st["kernel_launches"], st["graph"]))
        return out

    graph, host = run(False), run(True)
    assert [g[:3] for g in graph] == [h[:3] for h in host]
    assert graph[8][3] == 1 and host[8][3] == 0 and host[8][0] > 16


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
def test_solve(pd, prec):
    P = _problem(0)
    out = []
    for no_graph in (False, True):
        with pd.Plan.from_problem(P, precision=prec, no_graph=no_graph, eps_krylov=1e-5, **KW) as plan:
            _, st = plan.solve(torch.from_numpy(P.G).cuda(), allow_not_converged=True)
            out.append((st["refine_sweeps"], st["krylov_iters_total"], st["kernel_launches"]))
            assert st["graph"] == (0 if no_graph else 1)
    assert out[0] == out[1]
