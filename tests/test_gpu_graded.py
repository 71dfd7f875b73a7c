"""Operators whose off-diagonals are large against the diagonal (graded mass matrices, symmetrically scaled
operators): symmetric positive definite, not diagonally dominant, accepted by every plan.  Their row sums
say little about the pivots, so the binary32 loops must not eliminate from them.

Bounds.  Solutions in the norm in which the plan solves, ||M^{1/2} u||: the accuracy contract of the mixed
path, 1e-10, against the oracle, within the default number of sweeps, wherever the kernel that eliminates
from the diagonals (tune pint_rows) brings the refinement to convergence; with few time steps and masses
over twelve decades it does not.  One shifted solve in binary32 against
the same in binary64, relative 2-norm of each frequency: 8 u32 cond with cond <= 1 + 4 / (h^2 lambda_min),
the operator's own without the grading (symmetric scaling does not change the pivots' relative rounding)."""
import numpy as np
import pytest

import workloads as W
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


def _mass(n, ratio, seed):
    return np.exp((np.random.default_rng(seed).random(n) - 1.0) * np.log(ratio))


def _problem(n, nt, ratio, seed, T=1.0):
    P = W.with_mass(W.heat1d_forced(n, nt, T, seed=seed), seed=seed)
    P.m_diag[:] = _mass(n, ratio, seed)
    return P


def _scaled(P):
    """The same problem without a mass matrix: K' = M^{-1/2} K M^{-1/2}, unknown M^{1/2} u."""
    s = 1.0 / np.sqrt(P.m_diag)
    lo, up = P.k_lo.copy(), P.k_up.copy()
    lo[1:] *= s[1:] * s[:-1]
    up[:-1] *= s[1:] * s[:-1]
    return dict(k_lo=lo, k_diag=P.k_diag * s * s, k_up=up)


def _err(P, U, ref):
    m = np.sqrt(P.m_diag)
    return R.rel_err(U * m, ref * m)


@pytest.mark.parametrize("n,nt", [(40, 32), (300, 64), (1023, 128), (3000, 16)])
@pytest.mark.parametrize("ratio", [1e2, 1e4, 1e8, 1e12])
def test_graded_mass(pd, n, nt, ratio):
    P = _problem(n, nt, ratio, seed=n)
    G = torch.from_numpy(P.G).cuda()
    with pd.Plan.from_problem(P, precision="mixed", tune={"pint_rows": 8}) as plan:
        try:
            plan.solve(G)
        except pd.ParadiagError as e:
            assert e.status_name == "PD_ERR_NOT_CONVERGED" and (ratio, nt) == (1e12, 16)
            pytest.skip("not solved from the diagonals either")
    with pd.Plan.from_problem(P, precision="mixed") as plan:
        U, st = plan.solve(G)
    assert _err(P, U.cpu().numpy(), R.be_solve_refined(P)) <= 1e-10, st


def test_swapping_graded_operators_in_and_out(pd):
    """One plan, one pair of buffers (so one captured graph would serve all): uniform, graded, uniform."""
    probs = [_problem(255, 64, r, seed=5) for r in (1.0, 1e10, 1.0)]
    with pd.Plan.from_problem(probs[0], precision="mixed") as plan:
        G, U = torch.from_numpy(probs[0].G).cuda(), torch.empty((64, 255), dtype=torch.float64, device="cuda")
        sweeps = []
        for P in probs:
            plan.set_operator(tau=P.tau, k_lo=P.k_lo, k_diag=P.k_diag, k_up=P.k_up, m_diag=P.m_diag)
            G.copy_(torch.from_numpy(P.G))
            _, st = plan.solve(G, U)
            sweeps.append(st["refine_sweeps"])
            assert _err(P, U.cpu().numpy(), R.be_solve_refined(P)) <= 1e-10, st
    assert sweeps[0] == sweeps[2]


@pytest.mark.parametrize("alpha", [1.0, 1e-2])
def test_a_graded_problem_in_a_batch(pd, alpha):
    probs = [W.heat1d_forced(200, 64, seed=1), _problem(255, 64, 1e10, seed=2), W.advdiff1d_pulse(256, 64, seed=3)]
    with pd.Plan.from_problems(probs, precision="mixed", alpha=alpha) as plan:
        U, st = plan.solve(torch.from_numpy(plan.stack([P.G for P in probs])).cuda())
        parts = plan.unstack(U.cpu().numpy(), [P.nx for P in probs])
    for P, A in zip(probs, parts):
        ref = R.be_solve_refined(P)
        err = _err(P, A, ref) if P.m_diag is not None else R.rel_err(A, ref)
        assert err <= 1e-10, (P.name, st)


@pytest.mark.parametrize("ny", [1, 15])
def test_shifted_solves_against_binary64(pd, ny):
    n, nt = 127, 64
    P = _problem(n, nt, 1e8, seed=7)
    kw = dict(dim=1 if ny == 1 else 2, nx=n, nt=nt, tau=1.0 / nt, **_scaled(P))
    if ny > 1:
        ly, dy, uy = W.heat1d_operator(ny)
        kw.update(ny=ny, k_lo_y=ly, k_diag_y=dy, k_up_y=uy)
    gen = torch.Generator("cuda").manual_seed(ny)
    Rh = torch.randn((nt // 2 + 1, n * ny, 2), dtype=torch.float32, device="cuda", generator=gen)
    out = []
    for prec in ("mixed", "fp64"):
        with pd.Plan(precision=prec, **kw) as plan:
            X = torch.view_as_complex(Rh).to(plan.spectrum_dtype)
            out.append(plan.shifted_solve(X)[0].to(torch.complex128))
    err = float(((out[0] - out[1]).norm(dim=1) / out[1].norm(dim=1)).max())
    cond = 1.0 + 4.0 * (n + 1) ** 2 / np.pi ** 2
    assert err <= 8 * 2.0 ** -24 * cond
