"""The time DFTs in two register passes (csrc/rfft.cuh): every length from 32 to 2048 (and the first
ones outside, which stay with the general kernel), column counts at the edges of the narrow and wide
tiles, both precisions, row weights (alpha < 1), batches, and the modes of the inverse.

Tolerance, relative 2-norm: 3 u per radix-2 level, 3 log2(n) u (u = 2^-24 or 2^-53), for each of the
transform and, in binary32, the conversion of its input (one more u)."""
import numpy as np
import pytest

import workloads as W
from oracle import reference as R

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

UNIT = {"mixed": 2.0 ** -24, "fp64": 2.0 ** -53}


@pytest.fixture(scope="module")
def pd():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as entry

    entry.build()
    import paper_2304_12597_gb300 as pkg

    return pkg


def _plan(pd, prec, nt, ncols):
    """A plan of ncols columns: one 1D problem, or a batch of blocks of 500."""
    if ncols <= 4096:
        lo, di, up = W.heat1d_operator(ncols)
        return pd.Plan(dim=1, nx=ncols, nt=nt, tau=1e-3, k_lo=lo, k_diag=di, k_up=up, precision=prec)
    n, b = 500, ncols // 500
    lo, di, up = W.heat1d_operator(n)
    t = lambda a: np.tile(a, b)  # noqa: E731
    return pd.Plan(dim=1, nx=n, nt=nt, tau=1e-3, k_lo=t(lo), k_diag=t(di), k_up=t(up), precision=prec, batch=b)


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("ncols", [1, 7, 33, 1000, 10500])
@pytest.mark.parametrize("nt", [16, 32, 64, 128, 256, 512, 1024, 2048, 4096])
def test_transforms_match_definition(pd, nt, ncols, prec):
    if nt * ncols > 11e6:
        ncols = 2500  # (a wide tile for the long lengths)
    gen = torch.Generator("cuda").manual_seed(nt + ncols)
    tol = (3 * np.log2(nt) + 1) * UNIT[prec]
    with _plan(pd, prec, nt, ncols) as plan:
        X = torch.randn((nt, ncols), dtype=torch.float64, device="cuda", generator=gen)
        Xh = plan.time_dft(X)
        ref = torch.fft.rfft(X, dim=0)
        assert float((Xh - ref).abs().norm() / ref.abs().norm()) < tol
        # the inverse of any half spectrum: Re, so the imaginary parts at 0 and n/2 do not count
        Y = torch.randn((nt // 2 + 1, ncols, 2), dtype=torch.float64, device="cuda", generator=gen)
        Y = torch.view_as_complex(Y).to(plan.spectrum_dtype)
        Z = Y.to(torch.complex128)
        Z[0].imag.zero_()
        Z[-1].imag.zero_()
        want = torch.fft.irfft(Z, n=nt, dim=0)
        got = plan.time_idft(Y)
        assert float((got - want).norm() / want.norm()) < tol


@pytest.mark.parametrize("alpha", [1.0, 1e-4])
@pytest.mark.parametrize("nt", [32, 128, 512, 2048])
def test_solves_agree_with_the_general_kernel(pd, nt, alpha):
    """Refinement sweeps (U += delta), row weights, a batch with its per-problem norms and scales."""
    probs = [W.heat1d_forced(n, nt, 1.0, seed=n) for n in (60, 301)]
    G1 = torch.from_numpy(probs[1].G).cuda()
    for tune in ({}, {"fft_radix": 16}):
        for prec, tol in (("mixed", 1e-10), ("fp64", 1e-12)):
            with pd.Plan.from_problem(probs[1], precision=prec, alpha=alpha, tune=tune) as plan:
                got = plan.solve(G1)[0].cpu().numpy()
            assert R.rel_err(got, R.be_solve_refined(probs[1])) < tol
        with pd.Plan.from_problems(probs, precision="mixed", alpha=alpha, tune=tune) as plan:
            Uo, _ = plan.solve(torch.from_numpy(plan.stack([P.G for P in probs])).cuda())
            for P, A in zip(probs, plan.unstack(Uo.cpu().numpy(), [P.nx for P in probs])):
                assert R.rel_err(A, R.be_solve(P)) < 1e-10
