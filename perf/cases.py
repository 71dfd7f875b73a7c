"""The solves this framework is used for, as measurable cases.

A case is one call sequence a user's program makes on a plan it keeps:

  solve    Plan.solve on device arrays: a single problem, or a batch of problems in one plan
  host     Plan.solve_host: the right-hand side from pinned host memory, the solution back to it
  request  what the solve service does for one large request: swap its operator into a kept plan of
           the shape (Plan.set_operator), then Plan.solve
  advance  what the solve service does for a batch: swap the requests' operators into a kept batched
           plan (Plan.set_problems), then Plan.advance sweep by sweep until every problem converged

The problems are the repository's workloads (1D heat, 1D advection-diffusion with upwinding, 2D heat)
with seeded right-hand sides.  `exact` steps backward Euler in binary64: in the sine basis, where the
heat operators are diagonal, and with the dense inverse of I + tau K for advection-diffusion.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2304_12597_gb300 import Plan

PI = math.pi


def _case(name, path, kind, nx, nt, precision, *, ny=1, alpha=1.0, nu=1.0, T=1.0, batch=1, ragged=False, rhs="forced"):
    c = dict(path=path, kind=kind, nx=nx, ny=ny, nt=nt, precision=precision, alpha=alpha, nu=nu, T=T, batch=batch,
             ragged=ragged, rhs=rhs)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: one short 1D heat problem in binary64, bound by launches and latency
        _case("heat1d_127x64_fp64", "solve", "heat1d", 127, 64, "fp64", rhs="initial"),
        # the ordinary single 1D problem, forced heat, on both precision paths
        _case("heat1d_1023x1024_mixed", "solve", "heat1d", 1023, 1024, "mixed"),
        _case("heat1d_1023x1024_fp64", "solve", "heat1d", 1023, 1024, "fp64"),
        # the large single 1D problem: nonsymmetric operator, a pulse carried by advection
        _case("advdiff1d_4095x2048_mixed", "solve", "advdiff1d", 4095, 2048, "mixed", nu=1e-3, rhs="initial"),
        _case("advdiff1d_4095x2048_fp64", "solve", "advdiff1d", 4095, 2048, "fp64", nu=1e-3, rhs="initial"),
        # the headline: 2D heat, a smooth initial field, on both precision paths, and the mixed path
        # end to end from host buffers
        _case("heat2d_255x255x256_mixed", "solve", "heat2d", 255, 256, "mixed", ny=255, T=0.1, rhs="initial"),
        _case("heat2d_255x255x256_fp64", "solve", "heat2d", 255, 256, "fp64", ny=255, T=0.1, rhs="initial"),
        _case("heat2d_255x255x256_host", "host", "heat2d", 255, 256, "mixed", ny=255, T=0.1, rhs="initial"),
        # throughput: 32 independent problems in one plan
        _case("batch32_heat1d_1023x1024", "solve", "heat1d", 1023, 1024, "mixed", batch=32),
        # the service's 1D batch: heat and advection-diffusion requests of uneven n_x share a plan
        _case("serve_1d_8x2048x256", "advance", "mix1d", 2048, 256, "mixed", alpha=1e-4, nu=1e-2, batch=8, ragged=True),
        # the service's small-grid 2D batch
        _case("serve_2d_8x63x63x128", "advance", "heat2d", 63, 128, "mixed", ny=63, alpha=1e-4, nu=1e-2, batch=8),
        # the service's larger 2D request, alone in its plan
        _case("serve_2d_127x127x512", "request", "heat2d", 127, 512, "mixed", ny=127, alpha=1e-4, nu=1e-2),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case of the ranges above: n_x 31..4095 (2D: 31..255 by a side in {63, 127, 255}), n_t a
    power of two in 32..2048, both precisions, alpha = 1 and 1e-4, diffusion as each supports it."""
    what = rng.choice(("solve1d", "solve1d", "solve2d", "batch", "serve1d", "serve2d", "request"))
    precision = rng.choice(("mixed", "mixed", "fp64"))
    if what == "solve1d":
        kind, rhs = rng.choice(("heat1d", "advdiff1d")), rng.choice(("forced", "initial"))
        # forced advection-diffusion is Algorithm 3's ground: at alpha = 1 its inner system is ill-conditioned
        alpha = 1e-4 if (kind, rhs) == ("advdiff1d", "forced") else rng.choice((1.0, 1e-4))
        lo = -4.0 if alpha < 1.0 else (-1.0 if kind == "heat1d" else -3.0)
        return _case(None, "solve", kind, _log_int(rng, 31, 4095), 2 ** rng.randint(5, 11), precision, alpha=alpha,
                     nu=round(10.0 ** rng.uniform(lo, 0.0 if kind == "heat1d" else -1.0), 5), rhs=rhs)
    if what in ("solve2d", "request"):
        nx, ny = _log_int(rng, 31, 255), rng.choice((63, 127, 255))
        nt = 2 ** rng.randint(5, 11)
        while nx * ny * nt > 255 * 255 * 256:
            nt //= 2
        if what == "request":
            return _case(None, "request", "heat2d", ny, min(nt, 512), "mixed", ny=ny, alpha=1e-4,
                         nu=round(10.0 ** rng.uniform(-4.0, 0.0), 5))
        return _case(None, rng.choice(("solve", "solve", "host")), "heat2d", nx, nt, precision, ny=ny, T=0.1,
                     nu=round(10.0 ** rng.uniform(-0.5, 0.5), 3), rhs="initial")
    if what == "batch":
        batch, nx = rng.randint(2, 32), _log_int(rng, 127, 1023)
        return _case(None, "solve", "heat1d", nx, 2 ** rng.randint(5, 10), "mixed", batch=batch)
    nt = 2 ** rng.randint(5, 9)
    nu = round(10.0 ** rng.uniform(-4.0, 0.0), 5)
    if what == "serve1d":
        return _case(None, "advance", "mix1d", rng.choice((128, 256, 512, 1024, 2048, 4096)), nt, "mixed", alpha=1e-4,
                     nu=nu, batch=2 ** rng.randint(1, 4), ragged=True)
    return _case(None, "advance", "heat2d", 63, nt, "mixed", ny=63, alpha=1e-4, nu=nu, batch=2 ** rng.randint(1, 4))


# ---- the problems ---------------------------------------------------------------------------


def _problem_list(case, seed):
    """(kind, n_x, nu, generator seed) of each problem of the case."""
    rng = np.random.default_rng(seed)
    out = []
    for b in range(case["batch"]):
        kind = case["kind"] if case["kind"] != "mix1d" else ("heat1d", "advdiff1d")[b % 2]
        nx = case["nx"]
        if case["ragged"]:  # a size class of the service: more than half the slot
            nx = int(rng.integers(case["nx"] // 2 + 1, min(case["nx"], 4095) + 1))
        # the requests of one batch have diffusion coefficients of their own
        nu = case["nu"] if case["path"] == "solve" or case["path"] == "host" else case["nu"] * float(rng.uniform(0.5, 1.0))
        out.append((kind, nx, nu, int(rng.integers(1 << 31))))
    return out


def _axis(kind, n, nu):
    """(lo, diag, up) of nu tridiag(-1, 2, -1) / h^2, for advection-diffusion plus upwinding with a = 1."""
    h = 1.0 / (n + 1)
    d, a = nu / (h * h), (1.0 / h if kind == "advdiff1d" else 0.0)
    lo, di, up = np.full(n, -d - a), np.full(n, 2.0 * d + a), np.full(n, -d)
    lo[0] = up[-1] = 0.0
    return lo, di, up


def _operators(case, probs):
    out = []
    for kind, nx, nu, _ in probs:
        lo, di, up = _axis(kind, nx, nu)
        P = SimpleNamespace(dim=2 if kind == "heat2d" else 1, nx=nx, ny=case["ny"], nt=case["nt"],
                            tau=case["T"] / case["nt"], k_lo=lo, k_diag=di, k_up=up, k_lo_y=None, k_diag_y=None,
                            k_up_y=None, m_diag=None)
        if P.dim == 2:
            P.k_lo_y, P.k_diag_y, P.k_up_y = _axis(kind, case["ny"], nu)
        out.append(P)
    return out


def _sines(n, modes, device):
    x = torch.arange(1, n + 1, dtype=torch.float64, device=device) / (n + 1)
    return torch.sin(PI * torch.as_tensor(modes, dtype=torch.float64, device=device)[:, None] * x[None, :])


def _rhs(case, prob, out):
    """The right-hand side of one problem into out (n_t, n_x n_y): 16 space-time sine modes with N(0, 1)
    amplitudes ("forced"), or an initial value in the first row ("initial")."""
    kind, nx, _, seed = prob
    rng = np.random.default_rng(seed)
    dev, nt, ny = out.device, case["nt"], case["ny"]
    tau = case["T"] / nt
    if case["rhs"] == "forced":
        amp = torch.as_tensor(rng.standard_normal(16), device=dev)
        sp = _sines(nx, rng.integers(1, min(64, nx) + 1, 16), dev)
        if kind == "heat2d":
            sy = _sines(ny, rng.integers(1, min(64, ny) + 1, 16), dev)
            sp = (sy[:, :, None] * sp[:, None, :]).reshape(16, ny * nx)
        t = tau * torch.arange(1, nt + 1, dtype=torch.float64, device=dev)
        p = torch.as_tensor(rng.integers(1, 17, 16), dtype=torch.float64, device=dev)
        out.copy_((tau * torch.sin(PI * t[:, None] * p[None, :])) @ (amp[:, None] * sp))
        return
    out.zero_()
    if kind == "heat2d":
        m = min(32, nx, ny)
        k = np.arange(1, m + 1)
        coef = torch.as_tensor(rng.standard_normal((m, m)) / (k[:, None] ** 2 + k[None, :] ** 2), device=dev)
        out[0] = (_sines(ny, k, dev).T @ coef @ _sines(nx, k, dev)).reshape(-1)
    elif kind == "heat1d":
        k = np.concatenate([[1], rng.choice(np.arange(2, min(32, nx) + 1), min(8, nx - 1), replace=False)])
        amp = np.concatenate([[1.0], 0.1 * rng.standard_normal(len(k) - 1)])
        out[0] = torch.as_tensor(amp, device=dev) @ _sines(nx, k, dev)
    else:
        x = torch.arange(1, nx + 1, dtype=torch.float64, device=dev) / (nx + 1)
        out[0] = torch.exp(-((x - 0.25 - 0.1 * rng.random()) ** 2) / (2 * 0.05 ** 2))
        out[0] += torch.as_tensor(1e-3 * rng.standard_normal(nx), device=dev)


def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    probs = _problem_list(case, seed)
    ops = _operators(case, probs)
    kw = dict(precision=case["precision"], alpha=case["alpha"], device=dev)
    if case["batch"] > 1:
        plan = Plan.from_problems(ops, nx=case["nx"], **kw)
    else:
        plan = Plan.from_problem(ops[0], host_io=case["path"] == "host", **kw)
    G = torch.zeros((plan.nt, plan.nbar), dtype=torch.float64, device=dev)
    Gv = G.view(plan.nt, plan.batch, plan.slot)
    for b, prob in enumerate(probs):
        _rhs(case, prob, Gv[:, b, : prob[1] * case["ny"]])
    if case["path"] == "host":
        G = G.cpu().pin_memory()
        U = torch.empty_like(G).pin_memory()
    else:
        U = torch.empty_like(G)
    return SimpleNamespace(case=case, plan=plan, ops=ops, G=G, U=U)


def run(state):
    plan, G, U = state.plan, state.G, state.U
    path = state.case["path"]
    if path == "solve":
        return plan.solve(G, U)[0]
    if path == "host":
        return plan.solve_host(G, U)[0]
    if path == "request":
        P = state.ops[0]
        plan.set_operator(tau=P.tau, k_lo=P.k_lo, k_diag=P.k_diag, k_up=P.k_up, k_lo_y=P.k_lo_y, k_diag_y=P.k_diag_y,
                          k_up_y=P.k_up_y)
        return plan.solve(G, U)[0]
    plan.set_problems(state.ops)
    done, _ = plan.advance(G, U, [1] * plan.batch, steps=1)
    while 0 in done:
        done, _ = plan.advance(G, U, [0] * plan.batch, steps=1)
    return U


def work(case):
    """Right-hand side in and solution out, once; one Algorithm-1 solve's arithmetic (two real DFTs along
    time, three passes of n_t / 2 complex tridiagonal solves, in 2D two sine transforms along y)."""
    n = float(case["batch"] * case["nx"] * case["ny"] * case["nt"])
    flops = 5.0 * math.log2(case["nt"]) + 3 * 0.5 * 30.0
    if case["ny"] > 1:
        flops += 5.0 * math.log2(case["ny"] + 1)
    return {"bytes": 16.0 * n, "flops": flops * n}


# ---- the same solutions in plain torch, binary64 ----------------------------------------------


def _sine_matrix(n, device):
    return _sines(n, np.arange(1, n + 1), device) * math.sqrt(2.0 / (n + 1))  # orthonormal, symmetric


def _heat_eig(n, nu, device):
    j = torch.arange(1, n + 1, dtype=torch.float64, device=device)
    return 4.0 * nu * (n + 1) ** 2 * torch.sin(0.5 * PI * j / (n + 1)) ** 2


def _exact_one(case, prob, G, U):
    """Backward Euler u_j = (I + tau K)^{-1} (u_{j-1} + G_j) of one problem, G and U (n_t, n_x n_y)."""
    kind, nx, nu, _ = prob
    dev, nt, ny = G.device, case["nt"], case["ny"]
    tau = case["T"] / nt
    if kind == "advdiff1d":
        lo, di, up = (torch.as_tensor(a, device=dev) for a in _axis(kind, nx, nu))
        A = torch.diag(1.0 + tau * di) + torch.diag(tau * lo[1:], -1) + torch.diag(tau * up[:-1], 1)
        Ainv = torch.linalg.inv(A)
        u = torch.zeros(nx, dtype=torch.float64, device=dev)
        for j in range(nt):
            u = Ainv @ (u + G[j])
            U[j] = u
        return
    Sx = _sine_matrix(nx, dev)
    fac = _heat_eig(nx, nu, dev)
    W = G.reshape(nt, ny, nx) @ Sx
    if kind == "heat2d":
        Sy = _sine_matrix(ny, dev)
        W = torch.matmul(Sy, W)
        fac = _heat_eig(ny, nu, dev)[:, None] + fac[None, :]
    fac = 1.0 / (1.0 + tau * fac)
    u = torch.zeros_like(W[0])
    for j in range(nt):
        u = (u + W[j]) * fac
        W[j] = u
    if kind == "heat2d":
        W = torch.matmul(Sy, W)
    U.copy_((W @ Sx).reshape(nt, ny * nx))


def exact(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    probs = _problem_list(case, seed)
    nt, slot = case["nt"], case["nx"] * case["ny"]
    U = torch.zeros((nt, case["batch"], slot), dtype=torch.float64, device=dev)
    for b, prob in enumerate(probs):
        n = prob[1] * case["ny"]
        G = torch.empty((nt, n), dtype=torch.float64, device=dev)
        _rhs(case, prob, G)
        _exact_one(case, prob, G, U[:, b, :n])
    U = U.reshape(nt, case["batch"] * slot)
    return U.cpu() if case["path"] == "host" else U
