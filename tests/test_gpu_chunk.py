"""The binary32 shifted solves with chunks in registers (csrc/pint_chunk.cu), at the edges of
its teams: rows per block around 8 / 16 rows per lane times 8 .. 256 lanes, one and several
blocks, few and many frequencies.

Tolerance: the normwise backward error of each shifted system.  Row-wise diagonally dominant
systems are eliminated without growth (the multipliers and the chunks' couplings are at most
one), so the error is the rounding of the operations a row passes through: at most 8 complex
operations in its chunk and 6 in each of at most 8 cyclic-reduction levels, each within 3 u of
its result (u = 2^-24): 170 u.
"""
import numpy as np
import pytest

import workloads as W
from oracle import reference as R

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U32 = 2.0 ** -24
BOUND = 170 * U32


@pytest.fixture(scope="module")
def pd():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as entry

    entry.build()
    import paper_2304_12597_gb300 as pkg

    return pkg


def _check(plan, probs, slot):
    nt, nf = plan.nt, plan.nt // 2 + 1 if plan.nt > 1 else 1
    rng = np.random.default_rng(7)
    Rk = (rng.standard_normal((nf, plan.nbar)) + 1j * rng.standard_normal((nf, plan.nbar))).astype(np.complex64)
    Y, b = plan.shifted_solve(torch.from_numpy(Rk).cuda())
    Y, b = Y.cpu().numpy().astype(np.complex128), b.cpu().numpy()
    pi, gamma = R.circulant_eigs(nt)
    for i, P in enumerate(probs):
        c = slice(i * slot, i * slot + P.nx)
        y, r = Y[:, c], Rk[:, c].astype(np.complex128)
        # the coefficients the kernel holds: tau K rounded to binary32
        lo, di, up = [(P.tau * a).astype(np.float32).astype(np.float64) for a in (P.k_lo, P.k_diag, P.k_up)]
        s = (1.0 - pi[:nf])[:, None]
        Ay = (s + di) * y
        Ay[:, 1:] += lo[1:] * y[:, :-1]
        Ay[:, :-1] += up[:-1] * y[:, 1:]
        scale = np.max(np.abs(s + di) + np.abs(lo) + np.abs(up), axis=1) * np.linalg.norm(y, axis=1) + np.linalg.norm(r, axis=1)
        bw = np.linalg.norm(Ay - r, axis=1) / scale
        assert np.all(bw < BOUND), (P.nx, nt, float(bw.max()))
        w = np.where((np.arange(nf) == 0) | (2 * np.arange(nf) == nt), 1.0, 2.0)[:, None] * gamma[:nf, None]
        terms = (w * y).real
        assert np.all(np.abs(b[c] - terms.sum(0)) <= (nf + 4) * U32 * np.abs(w * y).sum(0)), (P.nx, nt)


@pytest.mark.parametrize("nt", [1, 2, 32, 256])
@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 63, 64, 65, 127, 128, 129, 255, 256, 257, 511, 512, 513, 1024, 1025, 2048,
                               2049, 4095, 4096])
def test_one_block(pd, n, nt):
    P = W.random_tridiag_problem(n, nt, seed=n + nt)
    with pd.Plan.from_problem(P, precision="mixed", tune={"zero_lane": -1}) as plan:
        _check(plan, [P], n)


@pytest.mark.parametrize("slot,nt", [(20, 64), (64, 16), (130, 256), (300, 32), (700, 8)])
def test_several_blocks(pd, slot, nt):
    probs = [W.random_tridiag_problem(n, nt, seed=n) for n in (slot, 1, slot // 2, slot - 1, 3)]
    with pd.Plan.from_problems(probs, precision="mixed", tune={"zero_lane": -1}) as plan:
        _check(plan, probs, slot)


@pytest.mark.parametrize("n", [5, 64, 200, 511, 1100, 3000])
def test_agrees_with_the_general_kernel(pd, n):
    """The same solve (several Algorithm-2 steps, final loops with x_m) through k_pint."""
    P = W.random_tridiag_problem(n, 64, seed=n)
    G = torch.from_numpy(P.G).cuda()
    out = []
    for tune in ({"zero_lane": -1}, {"zero_lane": -1, "pint_rows": 8}):
        for final in (0, -1):
            with pd.Plan.from_problem(P, precision="mixed", tune={**tune, "final_loop": final}) as plan:
                out.append(plan.solve(G)[0])
    ref = R.be_solve(P)
    for Uo in out:
        assert R.rel_err(Uo.cpu().numpy(), ref) < 1e-10


@pytest.mark.parametrize("make", [W.heat1d_operator, lambda n: W.advdiff1d_operator(n, 1.0, 1e-3)], ids=["heat", "upwind"])
@pytest.mark.parametrize("n", [40, 127, 255, 1023, 4095])
def test_zero_frequency_of_an_m_matrix_is_solved_to_working_accuracy(pd, n, make):
    """tau K itself (k = 0, condition up to 1e7) with a nonnegative right-hand side: the excess
    elimination adds terms of one sign only, so every entry keeps a relative error of the
    operations it passes through, at most 16 rows x 6 + 8 levels x 10 roundings of u each, and as
    many again on the way back: 400 u, whatever the condition."""
    lo, di, up = make(n)
    nt = 16
    with pd.Plan(dim=1, nx=n, nt=nt, tau=1.0 / nt, k_lo=lo, k_diag=di, k_up=up, precision="mixed",
                 tune={"zero_lane": -1}) as plan:
        r = np.random.default_rng(n).uniform(0.0, 1.0, (nt // 2 + 1, n)).astype(np.complex64)
        y = plan.shifted_solve(torch.from_numpy(r).cuda())[0][0].cpu().numpy()
    # the couplings as the kernel holds them, the row sums exact: binary64 elimination of the
    # dense matrix is accurate to kappa 2^-53 < 1e-8
    l32, u32 = (lo / nt).astype(np.float32).astype(float), (up / nt).astype(np.float32).astype(float)
    e32 = (((di + lo) + up) / nt).astype(np.float32).astype(float)
    A = np.diag(e32 - l32 - u32) + np.diag(l32[1:], -1) + np.diag(u32[:-1], 1)
    ref = np.linalg.solve(A, r[0].real.astype(float))
    assert np.max(np.abs(y.real - ref) / np.abs(ref)) < 400 * U32
    assert np.max(np.abs(y.imag)) <= 400 * U32 * np.max(np.abs(ref))
