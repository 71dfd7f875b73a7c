"""paradiag_batch_advance as one captured graph (GPU, through the C ABI).

From its eighth consecutive call with one (U, steps) pair on, a batched plan runs the sweeps of
a call as one graph launch; it launches exactly the kernels of the host-driven loops, so states,
iterates and statistics are identical to those of a plan that never captures.
"""
import pytest

import workloads as W

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


def _problems(dim):
    if dim == 2:
        return [W.heat2d_smooth(15, 16, 0.1, seed=s) for s in (1, 2)]
    return [W.heat1d_forced(255, 64, seed=1), W.advdiff1d_pulse(200, 64, seed=2),
            W.random_tridiag_problem(33, 64, seed=4)]


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("dim", [1, 2])
def test_captured_advance_equals_host_driven_advance(pd, prec, dim):
    """Three rounds of joins over 27 calls; the steps change (host-driven again), a solve with
    another buffer and a swap of the operators come in between, and the iterate moves to another
    buffer."""
    probs = _problems(dim)
    dev = torch.device("cuda:0")

    def run(no_graph):
        out = []
        with pd.Plan.from_problems(probs, precision=prec, device=dev, no_graph=no_graph) as plan:
            G = torch.from_numpy(plan.stack([P.G for P in probs])).to(dev)
            U, V = torch.zeros_like(G), torch.zeros_like(G)
            for call in range(27):
                join = [int(call % 9 == b) for b in range(plan.batch)]
                if call == 12:
                    plan.solve(G)
                if call == 13 and dim == 1:
                    plan.set_problems(probs)
                buf = V if call >= 25 else U
                state, st = plan.advance(G, buf, join, steps=2 if call in (14, 15) else 1)
                out.append((list(state), st["refine_sweeps"], st["krylov_iters_total"], st["kernel_launches"],
                            st["graph"], buf.clone()))
        return out

    for call, (a, b) in enumerate(zip(run(False), run(True))):
        assert a[:4] == b[:4], call
        assert a[4] == (1 if 7 <= call <= 13 or 23 <= call <= 24 else 0) and b[4] == 0, call
        assert torch.equal(a[5], b[5]), call
