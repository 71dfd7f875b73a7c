"""The time DFT of the 1D FP64 residual in registers (csrc/rfft_res.cu): every length from 32 to 2048,
column counts at the edges of the narrow and the wide tiles, row weights (alpha < 1), one problem and
batches with their scales.

A refined solve converges to the root of the residual that it forms, so a wrong value anywhere shows
in the result: it must agree with the general kernel's (any first-stage radix chosen by the caller
selects that one) within the sum of the two paths' bars, 2e-10, relative 2-norm."""
import numpy as np
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


def _plan(pd, nt, ncols, alpha, tune):
    if ncols <= 4096:
        lo, di, up = W.heat1d_operator(ncols)
        return pd.Plan(dim=1, nx=ncols, nt=nt, tau=1e-3, k_lo=lo, k_diag=di, k_up=up, precision="mixed", alpha=alpha,
                       tune=tune)
    n, b = 500, ncols // 500
    lo, di, up = W.heat1d_operator(n)
    t = lambda a: np.tile(a, b)  # noqa: E731
    return pd.Plan(dim=1, nx=n, nt=nt, tau=1e-3, k_lo=t(lo), k_diag=t(di), k_up=t(up), precision="mixed", batch=b,
                   alpha=alpha, tune=tune)


@pytest.mark.parametrize("alpha", [1.0, 1e-4])
@pytest.mark.parametrize("ncols", [1, 7, 33, 1000, 10500])
@pytest.mark.parametrize("nt", [32, 64, 128, 256, 512, 1024, 2048])
def test_refined_solves_agree_with_the_general_kernel(pd, nt, ncols, alpha):
    if nt * ncols > 11e6:
        ncols = 2500  # (a wide tile for the long lengths)
    gen = torch.Generator("cuda").manual_seed(nt + ncols)
    G = torch.randn((nt, ncols), dtype=torch.float64, device="cuda", generator=gen)
    out = []
    for tune in ({}, {"fft_radix": 16}):
        with _plan(pd, nt, ncols, alpha, tune) as plan:
            U, st = plan.solve(G)
            assert st["refine_sweeps"] > 1
            out.append(U)
    assert float((out[0] - out[1]).norm() / out[1].norm()) < 2e-10
