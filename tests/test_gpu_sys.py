"""FP64 shifted solves with a thread per system (csrc/pint_sys.cu) against the general loop (selected
by asking for stored factors): ragged row counts, unsymmetric operators, more basis vectors than one
pass of dots takes, the final loop's solves (no linearity, alpha < 1, batches), and the stage entry point.

Tolerances, relative 2-norm.  Refined solves: each path meets the FP64 bar of 1e-12, so they agree within
2e-12.  One shifted solve: 10 n u cond(tau K), the zero frequency's, for each path; with n <= 64 rows and
cond <= 4 n^2 / 9 that is below 2e-10 in all."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GENERAL = {"pint_factor": 1}


@pytest.fixture(scope="module")
def pd():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as entry

    entry.build()
    import paper_2304_12597_gb300 as pkg

    return pkg


def _plan(pd, nx, ny, nt, tune=None, batch=1, advect=False, **kw):
    """2D: ny modes of nx rows; ny = 1: a batch of 1D problems of nx rows."""
    lo, di, up = W.advdiff1d_operator(nx, 1.0, 1e-2) if advect else W.heat1d_operator(nx)
    if ny == 1:
        t = lambda a: np.tile(a, batch)  # noqa: E731
        return pd.Plan(dim=1, nx=nx, nt=nt, tau=1e-3, k_lo=t(lo), k_diag=t(di), k_up=t(up), precision="fp64", batch=batch,
                       tune=tune, **kw)
    ly, dy, uy = W.heat1d_operator(ny)
    return pd.Plan(dim=2, nx=nx, ny=ny, nt=nt, tau=1e-3, k_lo=lo, k_diag=di, k_up=up, k_lo_y=ly, k_diag_y=dy, k_up_y=uy,
                   precision="fp64", tune=tune, **kw)


def _rand(plan, seed):
    gen = torch.Generator("cuda").manual_seed(seed)
    return torch.randn((plan.nt, plan.nbar), dtype=torch.float64, device="cuda", generator=gen)


def _close(a, b, tol):
    assert float((a - b).norm() / b.norm()) < tol


# (nx, ny, nt, batch): 14592 systems and more; 65 x 511 leaves a partial last warp, 4 rows one group of loads
SHAPES = [(64, 127, 512, 1), (33, 511, 128, 1), (5, 255, 256, 1), (4, 15, 4096, 1), (300, 1, 512, 80)]


@pytest.mark.parametrize("advect", [False, True])
@pytest.mark.parametrize("nx,ny,nt,batch", SHAPES)
def test_shifted_solves(pd, nx, ny, nt, batch, advect):
    if nx > 64:
        nx = 50
    out = []
    for tune in (None, GENERAL):
        with _plan(pd, nx, ny, nt, tune, batch, advect) as plan:
            gen = torch.Generator("cuda").manual_seed(nx + ny)
            R = torch.randn((nt // 2 + 1, plan.nbar, 2), dtype=torch.float64, device="cuda", generator=gen)
            R = torch.view_as_complex(R)
            Y, b = plan.shifted_solve(R)
            _, b1 = plan.shifted_solve(R, want_y=False)
            Y1, _ = plan.shifted_solve(R, want_b=False)
            assert torch.equal(b, b1) and torch.equal(Y, Y1)
            out.append((Y, b))
    _close(out[0][0], out[1][0], 2e-10)
    _close(out[0][1], out[1][1], 2e-10)


@pytest.mark.parametrize("kw", [{}, {"alpha": 1e-4}, {"eps_krylov": 1e-15, "maxit": 20}, {"q": 2}, {"no_graph": True}],
                         ids=["default", "alpha", "many_steps", "frozen", "host_loop"])
@pytest.mark.parametrize("nx,ny,nt,batch", SHAPES)
def test_solves(pd, nx, ny, nt, batch, kw):
    if batch > 1 and "q" in kw:
        pytest.skip("batches run q = 1")
    out = []
    for tune in (None, {"final_loop": -1}, GENERAL):
        with _plan(pd, nx, ny, nt, tune, batch, **kw) as plan:
            U, st = plan.solve(_rand(plan, nt + nx))
            out.append(U)
    _close(out[0], out[2], 2e-12)
    _close(out[1], out[2], 2e-12)
