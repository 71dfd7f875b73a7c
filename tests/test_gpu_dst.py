"""The DST along y over half of the odd extension (csrc/dst.cu): lengths 63, 127 and 255, widths at
which the 64-column tiles cut through time slabs, batches, and the FP64 residual as its input,
against the definition and against the general kernel (tune fft_radix).

Tolerances.  Binary64 transform, relative 2-norm: 6 log2(N2) roundings of the FFT of length
N2 = 2 (n_y + 1), plus 16 of the reference's own dot products (random-sign sums of 255 terms).
Solves: the accuracy contract of the mixed and FP64 paths.
"""
import numpy as np
import pytest

import workloads as W
from oracle import reference as R

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U64 = 2.0 ** -53


@pytest.fixture(scope="module")
def pd():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as entry

    entry.build()
    import paper_2304_12597_gb300 as pkg

    return pkg


def _problem(nx, ny, nt, seed):
    lo, di, up = W.heat1d_operator(nx)
    ylo, ydi, yup = W.heat1d_operator(ny)
    rng = np.random.default_rng(seed)
    T = 0.05
    G = np.zeros((nt, ny * nx))
    x, y = np.arange(1, nx + 1) / (nx + 1), np.arange(1, ny + 1) / (ny + 1)
    for k, l, a in zip(rng.integers(1, 6, 8), rng.integers(1, 6, 8), rng.standard_normal(8)):
        G[0] += a * np.outer(np.sin(l * np.pi * y), np.sin(k * np.pi * x)).reshape(-1)
    G[1:] = 1e-3 * rng.standard_normal((nt - 1, ny * nx))
    return W.Problem(name="p", dim=2, nx=nx, ny=ny, nt=nt, T=T, tau=T / nt, k_lo=lo, k_diag=di, k_up=up, G=G, seed=seed,
                     recipe="", k_lo_y=ylo, k_diag_y=ydi, k_up_y=yup)


@pytest.mark.parametrize("ny", [63, 127, 255])
@pytest.mark.parametrize("nx,nt", [(77, 128), (64, 256), (33, 512), (1, 8192), (255, 64)])
def test_transform_matches_definition(pd, nx, ny, nt):
    P = _problem(nx, ny, 2, 0)
    with pd.Plan(dim=2, nx=nx, ny=ny, nt=nt, tau=1e-3, k_lo=P.k_lo, k_diag=P.k_diag, k_up=P.k_up, k_lo_y=P.k_lo_y,
                 k_diag_y=P.k_diag_y, k_up_y=P.k_up_y, precision="fp64", tune={"pint_factor": -1}) as plan:
        X = torch.randn((nt, ny * nx), dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(nx))
        Y = plan.dst_y(X)
    j = np.arange(1, ny + 1)
    S = np.sin(np.pi * ((j[:, None] * j[None, :]) % (2 * (ny + 1))) / (ny + 1)) * np.sqrt(2.0 / (ny + 1))
    ref = torch.matmul(torch.from_numpy(S).cuda(), X.view(nt, ny, nx)).view(nt, ny * nx)
    assert float((Y - ref).norm() / ref.norm()) < (6 * np.log2(2 * (ny + 1)) + 16) * U64


@pytest.mark.parametrize("prec,tol", [("mixed", 1e-10), ("fp64", 1e-12)])
@pytest.mark.parametrize("nx,ny,nt", [(77, 63, 128), (5, 127, 2048), (41, 255, 256)])
def test_solve_agrees_with_the_general_kernel(pd, nx, ny, nt, prec, tol):
    P = _problem(nx, ny, nt, 3)
    G = torch.from_numpy(P.G).cuda()
    out = []
    for tune in ({}, {"fft_radix": 16 if prec == "mixed" else 4}):
        with pd.Plan.from_problem(P, precision=prec, tune=tune) as plan:
            out.append(plan.solve(G)[0].cpu().numpy())
    ref = R.be_solve_refined(P)
    for Uo in out:
        assert R.rel_err(Uo, ref) < tol


def test_batch_of_grids_agrees_with_the_oracle(pd):
    probs = [_problem(40, 63, nt, 10 + nt) for nt in (128, 64, 128)]
    with pd.Plan.from_problems(probs, precision="mixed") as plan:
        Uo, _ = plan.solve(torch.from_numpy(plan.stack([P.G for P in probs])).cuda())
        parts = plan.unstack(Uo.cpu().numpy(), [P.nx * P.ny for P in probs], [P.nt for P in probs])
    for P, A in zip(probs, parts):
        assert R.rel_err(A, R.be_solve(P)) < 1e-10
