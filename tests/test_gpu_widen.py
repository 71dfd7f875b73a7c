"""binary32 -> binary64 on the stores of the inverse transforms (f32_to_f64_bits, csrc/pd_common.cuh):
exact for every finite number, subnormals among them, as the hardware conversion is; NaN stays NaN.
Reference: numpy's conversion and ldexp, bit for bit (all results are normal numbers of binary64)."""
import ctypes

import numpy as np
import pytest

from native_build import compile_snippet

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SOURCE = r"""
template <bool BRANCH>
__global__ void k_widen(int n, const float *x, int k, double *a, double *b) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  a[i] = cvt<double, BRANCH>(x[i]);
  b[i] = slot_store<BRANCH>(x[i], k);
}
extern "C" int run_widen(int branch, int n, const float *x, int k, double *a, double *b) {
  if (branch)
    k_widen<true><<<(n + 255) / 256, 256>>>(n, x, k, a, b);
  else
    k_widen<false><<<(n + 255) / 256, 256>>>(n, x, k, a, b);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return compile_snippet(tmp_path_factory.mktemp("widen"), SOURCE)


@pytest.mark.parametrize("branch", [0, 1])
@pytest.mark.parametrize("k", [0, 1, -1, 137, -600, 640])
def test_every_kind_of_number(lib, k, branch):
    bits = np.concatenate([
        np.arange(0, 70), 0x7fffff - np.arange(70), 0x800000 + np.arange(70),          # zero, subnormals, first normals
        np.random.default_rng(1).integers(0, 0x800000, 4000),                          # subnormals
        np.random.default_rng(2).integers(0x800000, 0x7f800000, 4000), [0x7f7fffff],   # normals
    ]).astype(np.uint32)
    x = np.concatenate([bits, bits | np.uint32(0x80000000)]).view(np.float32)
    X = torch.from_numpy(x).cuda()
    a, b = (torch.empty(len(x), dtype=torch.float64, device="cuda") for _ in range(2))
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    assert lib.run_widen(branch, len(x), p(X), k, p(a), p(b)) == 0
    want = x.astype(np.float64)
    assert np.array_equal(a.cpu().numpy().view(np.int64), want.view(np.int64))
    assert np.array_equal(b.cpu().numpy().view(np.int64), np.ldexp(want, k).view(np.int64))


@pytest.mark.parametrize("branch", [0, 1])
def test_infinities_and_nan(lib, branch):
    X = torch.tensor([float("inf"), -float("inf"), float("nan")], dtype=torch.float32, device="cuda")
    a, b = (torch.empty(3, dtype=torch.float64, device="cuda") for _ in range(2))
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    assert lib.run_widen(branch, 3, p(X), 5, p(a), p(b)) == 0
    for t in (a.cpu(), b.cpu()):
        assert t[0] == float("inf") and t[1] == -float("inf") and torch.isnan(t[2])


def test_small_values_reach_the_solution():
    """The inverse time DFT of a binary32 plan: a constant column's half spectrum is its first row alone,
    n c, and the transform returns c, here below binary32's normal range."""
    import paper_2304_12597_gb300 as pkg

    n, nt = 40, 64
    c = np.ldexp(np.arange(1.0, n + 1), -140)
    with pkg.Plan(dim=1, nx=n, nt=nt, tau=1.0, k_lo=-np.ones(n), k_diag=np.full(n, 2.0), k_up=-np.ones(n),
                  precision="mixed") as plan:
        Y = torch.zeros((nt // 2 + 1, n), dtype=torch.complex64, device="cuda")
        Y[0] = torch.from_numpy(nt * c).to(torch.complex64)
        X = plan.time_idft(Y).cpu().numpy()
    assert np.array_equal(X, np.tile(c, (nt, 1)))
