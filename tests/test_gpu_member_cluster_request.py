"""A caller's krylov_cluster on a batched plan: the size asked for is the size taken, as for single problems
(0 still chooses, problems of fewer than 256 unknowns stay with one CTA), and the solutions meet the bars of
their precision (1e-10 mixed, 1e-12 FP64; two paths agree within twice that), also where the clusters of all
problems do not fit the SMs side by side."""
import pytest

import workloads as W
from native_build import compile_snippet

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SOURCE = r"""
extern "C" int cluster_size(int members, int len, int want) { return member_cluster_size(members, len, want); }
extern "C" int sms() { return sm_count(); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.zeros(1, device="cuda")
    return compile_snippet(tmp_path_factory.mktemp("cluster"), SOURCE)


@pytest.mark.parametrize("members", [2, 8, 60])
def test_the_size_asked_for(lib, members):
    for want in (4, 5, 8, 12, 16):
        assert lib.cluster_size(members, 256, want) == want
        assert lib.cluster_size(members, 255, want) == 0
    fits = [c for c in (8, 4) if c * members <= lib.sms()]
    assert lib.cluster_size(members, 4096, 0) == (fits[0] if fits else 0)


@pytest.mark.parametrize("prec,tol", [("mixed", 2e-10), ("fp64", 2e-12)])
@pytest.mark.parametrize("n,nt,batch", [(256, 16, 2), (2048, 32, 3), (300, 16, 45)])
def test_solutions(lib, n, nt, batch, prec, tol):
    import paper_2304_12597_gb300 as pkg

    make = [W.heat1d_forced, W.advdiff1d_pulse, W.random_tridiag_problem]
    probs = [make[i % 3](n - (i * 7) % 40, nt, seed=i) for i in range(batch)]
    out = []
    for want in (-1, 4, 5, 16):
        with pkg.Plan.from_problems(probs, precision=prec, tune={"krylov_cluster": want}) as plan:
            U, _ = plan.solve(torch.from_numpy(plan.stack([P.G for P in probs])).cuda())
            out.append([torch.from_numpy(a) for a in plan.unstack(U.cpu().numpy(), [P.nx for P in probs])])
    for other in out[1:]:
        for i, (a, b) in enumerate(zip(out[0], other)):
            assert float((a - b).norm() / a.norm()) < tol, i
