"""Shared memory of the persistent Algorithm-2 step (host arithmetic, no GPU): at m = 1 each of the CTA's 16
warps keeps its sums in a slice of (2 m^2 + 2 m) complex and m^2 real values (80 bytes), and every later step
needs at least one warp's slice and the solve's matrices."""
import ctypes

import pytest

import __graft_entry__ as entry


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    entry.build()
    from native_build import compile_snippet

    so = compile_snippet(tmp_path_factory.mktemp("smem"),
                         'extern "C" long long smem(int maxit, int nf, int elem) { return (long long)step_tail_smem(maxit, nf, elem); }')
    so.smem.restype = ctypes.c_longlong
    return so


@pytest.mark.parametrize("elem", [4, 8])
@pytest.mark.parametrize("maxit", [1, 2, 3, 8, 32])
def test_covers_every_step(lib, maxit, elem):
    for nf in (1, 9, 17, 129, 1025):
        have = lib.smem(maxit, nf, elem)
        assert have >= 16 * 80 and have >= nf * 2 * elem
        for m in range(1, maxit + 1):
            slice_bytes = ((2 * m * m + 2 * m) * 16 + m * m * 8 + 15) // 16 * 16
            assert have >= slice_bytes and have >= (2 * m * m + m) * 16 + (m + 1) * 8
