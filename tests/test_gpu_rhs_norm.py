"""The norms that the time DFTs of binary64 plans take.  Forward, of the input: binary64 squares, summed in
binary64 within a thread; across threads the sums are binary32 (csrc/pd_fft_tail.cuh).  Inverse, of the
output: squares of values rounded to nearest in binary32.

With every value 1 - 2^-50 a thread's sum is an integer but for less than 2^-24 of it, so binary32 holds it
exactly, and sums of 32 of them too: the norm is sqrt(n ncols) up to 2^-24 n_values roundings of the
binary64 additions and the values' own distance from one."""
import ctypes

import numpy as np
import pytest

from native_build import compile_snippet

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SOURCE = r"""
extern "C" int run_colsum(const double2 *S, int64_t ncols, int n, const double2 *tw, double *X, double *colsum) {
  Ctx c;
  int np = 0;
  launch_fft_c2r<double>(c, reinterpret_cast<const cpx<double> *>(S), ncols, ncols, n,
                         reinterpret_cast<const cpx<double> *>(tw), X, ncols, 0, nullptr, &np, nullptr, nullptr, colsum);
  return (int)cudaDeviceSynchronize();
}
extern "C" int run_norm(const double *X, int64_t ncols, int n, const double2 *tw, double2 *S, double *part, int *counter,
                        double *dst) {
  Ctx c;
  RhsNorm rn;
  rn.part = part;
  rn.counter = counter;
  rn.dst = dst;
  launch_fft_r2c<double, double>(c, X, ncols, ncols, n, reinterpret_cast<const cpx<double> *>(tw),
                                 reinterpret_cast<cpx<double> *>(S), ncols, nullptr, &rn);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return compile_snippet(tmp_path_factory.mktemp("norm"), SOURCE)


@pytest.mark.parametrize("n,ncols", [(32, 64), (64, 5000), (128, 96), (256, 20000), (512, 8192), (1024, 4096), (2048, 2048)])
def test_binary64_squares(lib, n, ncols):
    X = torch.full((n, ncols), 1.0 - 2.0 ** -50, dtype=torch.float64, device="cuda")
    k = np.arange(n // 2)
    tw = torch.from_numpy(np.exp(-2j * np.pi * k / n)).cuda()
    S = torch.empty((n // 2 + 1, ncols), dtype=torch.complex128, device="cuda")
    part = torch.zeros(ncols + 1024, dtype=torch.float64, device="cuda")
    counter = torch.zeros(1, dtype=torch.int32, device="cuda")
    dst = torch.zeros(1, dtype=torch.float64, device="cuda")
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    assert lib.run_norm(p(X), ctypes.c_int64(ncols), n, p(tw), p(S), p(part), p(counter), p(dst)) == 0
    want = np.sqrt(float(n * ncols))
    assert abs(float(dst[0]) - want) <= 1e-12 * want


@pytest.mark.parametrize("n,ncols", [(32, 64), (64, 5000), (128, 96), (256, 20000), (512, 8192), (1024, 4096), (2048, 2048)])
def test_squares_of_rounded_values(lib, n, ncols):
    """A column of 1 - 2^-26 everywhere (its spectrum is the first row alone): to nearest in binary32 that is
    one, so a column's sum of squares is n, exactly."""
    tw = torch.from_numpy(np.exp(-2j * np.pi * np.arange(n // 2) / n)).cuda()
    S = torch.zeros((n // 2 + 1, ncols), dtype=torch.complex128, device="cuda")
    S[0] = n * (1.0 - 2.0 ** -26)
    X = torch.empty((n, ncols), dtype=torch.float64, device="cuda")
    colsum = torch.zeros(ncols, dtype=torch.float64, device="cuda")
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    assert lib.run_colsum(p(S), ctypes.c_int64(ncols), n, p(tw), p(X), p(colsum)) == 0
    assert torch.allclose(X, torch.full_like(X, 1.0 - 2.0 ** -26), rtol=1e-14, atol=0.0)
    assert torch.equal(colsum, torch.full_like(colsum, float(n)))
