"""The batches' norms (csrc/batch.cu): every slot's sum of squares in binary64, and the exponents from it.

Bound: n values summed in any order, n 2^-53 relative (all terms are nonnegative)."""
import ctypes

import numpy as np
import pytest

from native_build import compile_snippet

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SOURCE = r"""
extern "C" int run_norms(const double *G, int64_t nt, int batch, int nxm, int nc, double *part, int *ex, int *zero,
                         const double **gslot) {
  Ctx c;
  launch_batch_exponents(c, G, nt, batch, nxm, nc, part, ex, zero, gslot);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return compile_snippet(tmp_path_factory.mktemp("norms"), SOURCE)


@pytest.mark.parametrize("nt,nxm", [(1, 1), (3, 31), (64, 33), (17, 255), (9, 257), (128, 1023), (32, 4096)])
@pytest.mark.parametrize("nc", [1, 5])
def test_sums_are_binary64(lib, nt, nxm, nc):
    mags = (1.0, 0.0, 1e-150, 1e150, 1e-170, 1.0)
    B = len(mags)
    rng = np.random.default_rng(nt + nxm)
    G = rng.standard_normal((nt, B, nxm)) * np.array(mags)[None, :, None]
    G[:, 5] = 1.0 - 2.0 ** -50  # values that binary32 would round or cut
    g = torch.from_numpy(G).cuda()
    part = torch.zeros((B, nc), dtype=torch.float64, device="cuda")
    ex, zero = (torch.full((B,), 77, dtype=torch.int32, device="cuda") for _ in range(2))
    gslot = torch.zeros(1, dtype=torch.int64, device="cuda")
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    assert lib.run_norms(p(g), ctypes.c_int64(nt), B, nxm, nc, p(part), p(ex), p(zero), p(gslot)) == 0
    assert int(gslot[0]) == g.data_ptr()
    s = part.sum(1).cpu().numpy()
    for b in range(B):
        ref = float(np.sum(np.square(np.longdouble(G[:, b]))).astype(np.float64)) if mags[b] > 1e-160 else 0.0
        assert abs(s[b] - ref) <= (nt * nxm + 2) * 2.0 ** -53 * ref, b
        assert int(zero[b]) == (ref == 0.0), b
        e2 = int(np.frexp(s[b])[1]) if ref else 0
        assert int(ex[b]) == -int(e2 / 2), b
