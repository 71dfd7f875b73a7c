"""The operator's device arrays (csrc/operator.cu) and the zero-frequency weight beside them: a
plan whose operator was swapped in solves exactly as a plan built with it, and the weight equals
its definition, for block counts around the eight blocks that are eliminated side by side."""
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


def _weight(P, nt, mus):
    """max_i |(l A_0)^{-1} (1, or (-1)^i)|_i over the blocks tau (K + mu I), alpha = 1."""
    worst = 0.0
    for mu in mus:
        A = P.tau * (np.diag(P.k_diag + mu) + np.diag(P.k_lo[1:], -1) + np.diag(P.k_up[:-1], 1))
        e = np.ones(P.nx)
        s = np.where(np.arange(P.nx) % 2, -1.0, 1.0)
        worst = max(worst, np.abs(np.linalg.solve(A, np.stack([e, s], 1))).max())
    return worst / nt


def _args(P):
    return dict(tau=P.tau, k_lo=P.k_lo, k_diag=P.k_diag, k_up=P.k_up, k_lo_y=P.k_lo_y, k_diag_y=P.k_diag_y,
                k_up_y=P.k_up_y, m_diag=P.m_diag)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("case", ["1d", "1d_mass", "2d_3", "2d_7", "2d_15"])
def test_swapped_operator_equals_built_operator(pd, prec, case):
    if case.startswith("2d"):
        n = int(case[3:])
        A, B = W.heat2d_smooth(n, 16, 0.5, seed=1), W.heat2d_smooth(n, 16, 0.3, seed=2)
        B.k_diag, B.k_lo, B.k_up = 1.5 * B.k_diag, 1.25 * B.k_lo, 1.25 * B.k_up
    else:
        A, B = W.random_tridiag_problem(67, 16, seed=1), W.random_tridiag_problem(67, 16, T=0.7, seed=2)
        if case == "1d_mass":
            A, B = W.with_mass(A, 1), W.with_mass(B, 2)
    G = torch.from_numpy(B.G).cuda()
    with pd.Plan.from_problem(B, precision=prec) as plan:
        want, st = plan.solve(G)
    with pd.Plan.from_problem(A, precision=prec) as plan:
        plan.set_operator(**_args(B))
        got, _ = plan.solve(G)
    assert torch.equal(got, want)
    if prec == "mixed" and case != "1d_mass":
        mus = [0.0]
        if case.startswith("2d"):
            mus = B.k_diag_y[0] + 2.0 * B.k_up_y[0] * np.cos(np.pi * np.arange(1, B.ny + 1) / (B.ny + 1))
        ref = _weight(B, B.nt, mus)
        # Thomas elimination of dominant blocks: a few roundings a row, and of K's condition
        assert abs(st["zero_freq_weight"] - ref) <= 1e-11 * ref


@pytest.mark.parametrize("count", [2, 8, 9])
@pytest.mark.parametrize("dim", [1, 2])
def test_swapped_batch_equals_built_batch(pd, dim, count):
    if dim == 1:
        mk = lambda s: [W.random_tridiag_problem(20 + 3 * b, 16, seed=s + b) for b in range(count)]  # noqa: E731
    else:
        mk = lambda s: [W.heat2d_smooth(7, 16, 0.1 + 0.05 * b, seed=s + b) for b in range(count)]  # noqa: E731
    A, B = mk(100), mk(200)
    with pd.Plan.from_problems(B, precision="mixed", nx=64) as plan:
        G = torch.from_numpy(plan.stack([P.G for P in B])).cuda()
        want, _ = plan.solve(G)
    with pd.Plan.from_problems(A, precision="mixed", nx=64) as plan:
        plan.set_problems(B)
        got, _ = plan.solve(G)
    assert torch.equal(got, want)
