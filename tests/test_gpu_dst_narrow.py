"""k_dst2 (csrc/dst.cu) on grids one and two columns wide: every lane of a tile is a slab of its own (or shares
it with one neighbour), and a tile's column pairs come from different problems.  The shapes lie above the
dispatch line, 64 columns per SM, which is checked.

Bounds as in test_gpu_dst: the binary64 transform against its definition, and solves to the precisions' bars
against the oracle."""
import numpy as np
import pytest

from test_gpu_dst import U64, _problem
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


def _above_the_line(plan):
    sms = torch.cuda.get_device_properties(plan.device).multi_processor_count
    return plan.batch * plan.nt * plan.nx >= 64 * sms


def _stack(plan, probs):
    return torch.from_numpy(plan.stack([P.G for P in probs])).cuda()


@pytest.mark.parametrize("ny", [63, 127, 255])
@pytest.mark.parametrize("nx,nt", [(1, 4096), (2, 2048)])
def test_transform(pd, nx, ny, nt):
    probs = [_problem(nx, ny, 2, s) for s in range(4)]
    cat = lambda f: np.concatenate([getattr(P, f) for P in probs])  # noqa: E731
    with pd.Plan(dim=2, nx=nx, ny=ny, nt=nt, tau=1e-3, k_lo=cat("k_lo"), k_diag=cat("k_diag"), k_up=cat("k_up"),
                 k_lo_y=cat("k_lo_y"), k_diag_y=cat("k_diag_y"), k_up_y=cat("k_up_y"), batch=4, precision="fp64") as plan:
        assert _above_the_line(plan)
        gen = torch.Generator("cuda").manual_seed(nx + ny)
        X = torch.randn((nt, plan.nbar), dtype=torch.float64, device="cuda", generator=gen)
        Y = plan.dst_y(X)
    j = np.arange(1, ny + 1)
    S = np.sin(np.pi * ((j[:, None] * j[None, :]) % (2 * (ny + 1))) / (ny + 1)) * np.sqrt(2.0 / (ny + 1))
    ref = torch.matmul(torch.from_numpy(S).cuda(), X.view(nt * 4, ny, nx)).view(nt, -1)
    assert float((Y - ref).norm() / ref.norm()) < (6 * np.log2(2 * (ny + 1)) + 16) * U64


@pytest.mark.parametrize("prec,ny,tol", [("mixed", 63, 1e-10), ("fp64", 63, 1e-12), ("fp64", 127, 1e-12)])
@pytest.mark.parametrize("nx,nt", [(1, 4096), (2, 2048)])
def test_solves(pd, nx, ny, nt, prec, tol):
    probs = [_problem(nx, ny, nt, 20 + s) for s in range(4)]
    with pd.Plan.from_problems(probs, precision=prec) as plan:
        assert _above_the_line(plan)
        U, st = plan.solve(_stack(plan, probs))
        assert st["refine_sweeps"] > 1  # the residual transform ran
        parts = plan.unstack(U.cpu().numpy(), [nx * ny] * 4)
    for P, A in zip(probs[:2], parts):
        assert R.rel_err(A, R.be_solve_refined(P)) < tol, st
