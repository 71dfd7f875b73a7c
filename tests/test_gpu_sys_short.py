"""FP64 shifted solves with a thread per system (csrc/pint_sys.cu) on the shortest blocks, 1 to 5 rows: less
than, exactly and more than the rows whose loads go out together.  The route is checked, not assumed: the
general loop sums b by its own reduction, this one by the column sum over the stored solutions.

Tolerances, relative 2-norm: one shifted solve, 10 n u cond(tau K) of the zero frequency for each path, with
cond <= 4 (n_y + 1)^2 + 4 (n + 1)^2 < 1.1e6 and n = 5 below 1.3e-8 in all; refined solves, twice the FP64
bar of 1e-12."""
import pytest

from test_gpu_sys import GENERAL, _close, _plan, _rand

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


# n_bar >= 256 (so that the vector steps run on a cluster and b is not reduced by Algorithm 2's start)
SHAPES = [(1, 511, 64), (2, 255, 256), (3, 255, 128), (4, 255, 256), (5, 255, 256)]


def _families(plan):
    return {k["name"]: k["launches"] for k in plan.kernel_times()}


@pytest.mark.parametrize("nx,ny,nt", SHAPES)
def test_short_blocks(pd, nx, ny, nt):
    Y, B, U = [], [], []
    for tune in (None, GENERAL):
        with _plan(pd, nx, ny, nt, tune) as plan:
            gen = torch.Generator("cuda").manual_seed(nx + ny)
            R = torch.randn((nt // 2 + 1, plan.nbar, 2), dtype=torch.float64, device="cuda", generator=gen)
            plan.set_timing(True)
            y, b = plan.shifted_solve(torch.view_as_complex(R))
            fam = _families(plan)
            assert ("zsum" in fam, "acc_reduce" in fam) == ((True, False) if tune is None else (False, True)), fam
            plan.set_timing(False)
            U.append(plan.solve(_rand(plan, nt + nx))[0])
            Y.append(y)
            B.append(b)
    _close(Y[0], Y[1], 1.3e-8)
    _close(B[0], B[1], 1.3e-8)
    _close(U[0], U[1], 2e-12)
