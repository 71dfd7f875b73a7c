"""The exact scaling of binary64 values on the batches' loads and stores (pow2_scale, csrc/pd_common.cuh):
x 2^k as ldexp gives it, with gradual underflow, subnormal inputs, infinities and NaN.
Reference: the C library's ldexp through numpy, bit for bit."""
import ctypes

import numpy as np
import pytest

import workloads as W
from native_build import compile_snippet

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SOURCE = r"""
__global__ void k_scale(int n, const double *x, int k, double *a, double *b) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  a[i] = slot_load<double>(x[i], k);
  b[i] = slot_store(x[i], k);
}
extern "C" int run_scale(int n, const double *x, int k, double *a, double *b) {
  k_scale<<<(n + 255) / 256, 256>>>(n, x, k, a, b);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return compile_snippet(tmp_path_factory.mktemp("scale"), SOURCE)


@pytest.mark.parametrize("k", [0, 1, -1, 52, -53, 500, -540, 640, -640])
def test_equals_ldexp(lib, k):
    rng = np.random.default_rng(3)
    top, one = 0x7ff0000000000000, 0x0010000000000000
    bits = np.concatenate([
        np.arange(70), one - 1 - np.arange(70), one + np.arange(70), top - 1 - np.arange(70), [top],
        rng.integers(0, one, 3000), rng.integers(one, top, 12000),
    ]).astype(np.uint64)
    # magnitudes around the lower end after the scaling
    edge = np.ldexp(1.0 + rng.random(4000), np.clip(rng.integers(-1080, -1015, 4000) - k, -1074, 1000))
    x = np.concatenate([bits, bits | np.uint64(1 << 63)]).view(np.float64)
    x = np.concatenate([x, edge, -edge])
    X = torch.from_numpy(x).cuda()
    a, b = (torch.empty(len(x), dtype=torch.float64, device="cuda") for _ in range(2))
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    assert lib.run_scale(len(x), p(X), k, p(a), p(b)) == 0
    with np.errstate(over="ignore", under="ignore"):
        want = np.ldexp(x, k).view(np.int64)
    assert np.array_equal(a.cpu().numpy().view(np.int64), want)
    assert np.array_equal(b.cpu().numpy().view(np.int64), want)


def test_subnormal_columns_of_a_problem():
    """A problem whose K is diagonal: its columns are independent recurrences.  Those whose right-hand side
    falls below 2^-1022 once the problem is scaled to unit norm (2^23) keep their solution, to the spacing of
    the scaled values (2^-1074 against 3e-308 2^-23: 1.4e-9) for some twenty roundings in each of 64 steps."""
    import paper_2304_12597_gb300 as pkg

    n, nt, tau, d = 64, 64, 0.25, 2.0
    P = W.random_tridiag_problem(n, nt, seed=1)
    z = np.zeros(n)
    prob = W.Problem(name="d", dim=1, nx=n, ny=1, nt=nt, T=nt * tau, tau=tau, k_lo=z, k_diag=np.full(n, d), k_up=z,
                     G=P.G, seed=0, recipe="")
    G = np.zeros((nt, n))
    G[:, 0] = 2.0 ** 20
    G[:, 32:] = 3e-308
    with pkg.Plan.from_problems([prob, prob], precision="fp64") as plan:
        U, _ = plan.solve(torch.from_numpy(plan.stack([G, G])).cuda())
        parts = plan.unstack(U.cpu().numpy(), [n, n])
    u = np.zeros(n)
    for t in range(nt):
        u = (u + G[t]) / (1.0 + tau * d)
        for A in parts:
            np.testing.assert_allclose(A[t, 32:], u[32:], rtol=2e-6)
            np.testing.assert_allclose(A[t, 0], u[0], rtol=1e-12)
