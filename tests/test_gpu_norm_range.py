"""The range of the norms that the binary32 time DFTs take: squares that fit binary32 in sums of 16 (inverse,
per thread) and of 1024 (forward, per warp), the most that the general transforms add there, must not
overflow in the register transforms either.

Columns of one value v; bound: 64 2^-24 relative for sums of up to 64 equal terms, rounded one by one."""
import ctypes

import numpy as np
import pytest

from native_build import compile_snippet

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SOURCE = r"""
extern "C" int run_colsum(const float2 *S, int64_t ncols, int n, const float2 *tw, double *X, double *colsum) {
  Ctx c;
  int np = 0;
  launch_fft_c2r<float>(c, reinterpret_cast<const cpx<float> *>(S), ncols, ncols, n,
                        reinterpret_cast<const cpx<float> *>(tw), X, ncols, 0, nullptr, &np, nullptr, nullptr, colsum);
  return (int)cudaDeviceSynchronize();
}
extern "C" int run_norm(const double *X, int64_t ncols, int n, const float2 *tw, float2 *S, double *part, int *counter,
                        double *dst) {
  Ctx c;
  RhsNorm rn;
  rn.part = part;
  rn.counter = counter;
  rn.dst = dst;
  launch_fft_r2c<float, double>(c, X, ncols, ncols, n, reinterpret_cast<const cpx<float> *>(tw),
                                reinterpret_cast<cpx<float> *>(S), ncols, nullptr, &rn);
  return (int)cudaDeviceSynchronize();
}
"""
SIZES = [(n, c) for n in (32, 64, 128, 256, 512, 1024, 2048) for c in (50, 12000)]
TOL = 64 * 2.0 ** -24


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return compile_snippet(tmp_path_factory.mktemp("range"), SOURCE)


def _p(t):
    return ctypes.c_void_p(t.data_ptr())


def _tw(n):
    return torch.from_numpy(np.exp(-2j * np.pi * np.arange(n // 2) / n).astype(np.complex64)).cuda()


@pytest.mark.parametrize("v", [4e18, 1.0, 1e-15])
@pytest.mark.parametrize("n,ncols", SIZES)
def test_inverse(lib, n, ncols, v):
    assert 16 * v * v < 3.4e38
    S = torch.zeros((n // 2 + 1, ncols), dtype=torch.complex64, device="cuda")
    S[0] = n * v
    X = torch.empty((n, ncols), dtype=torch.float64, device="cuda")
    colsum = torch.zeros(ncols, dtype=torch.float64, device="cuda")
    assert lib.run_colsum(_p(S), ctypes.c_int64(ncols), n, _p(_tw(n)), _p(X), _p(colsum)) == 0
    assert float((colsum / (n * v * v) - 1.0).abs().max()) < TOL


@pytest.mark.parametrize("v", [5e17, 1.0, 1e-15])
@pytest.mark.parametrize("n,ncols", SIZES)
def test_forward(lib, n, ncols, v):
    assert 1024 * v * v < 3.4e38
    X = torch.full((n, ncols), v, dtype=torch.float64, device="cuda")
    S = torch.empty((n // 2 + 1, ncols), dtype=torch.complex64, device="cuda")
    part = torch.zeros(ncols + 1024, dtype=torch.float64, device="cuda")
    counter = torch.zeros(1, dtype=torch.int32, device="cuda")
    dst = torch.zeros(1, dtype=torch.float64, device="cuda")
    assert lib.run_norm(_p(X), ctypes.c_int64(ncols), n, _p(_tw(n)), _p(S), _p(part), _p(counter), _p(dst)) == 0
    assert abs(float(dst[0]) / (np.sqrt(float(n * ncols)) * v) - 1.0) < TOL
