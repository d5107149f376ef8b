"""rick_workspace_size counts the two-pass transform's second plane buffer where
a handle takes it, and only there: not with grid correction by a kernel that
amplifies rounding too much, nor by request of another transform.  Against
cuFFT's 2D plan (RICK_FFT_2D, without it) the transform needs the buffer (8 n^2
bytes per plane, 16 planes) and two screen tables of a quarter plane each, 3 % of
it; twiddles, tile bits and row ranges are below 1 %."""
import ctypes

import pytest


@pytest.fixture(scope="module")
def lib():
    from paper_2504_00959_gb300 import build
    build.build()
    from paper_2504_00959_gb300 import _lib
    return _lib.load()


GAUSS, KB = 0, 1


@pytest.mark.parametrize("n", [1024, 2048, 4096])
@pytest.mark.parametrize("kernel,S,correct,flag,second", [
    (KB, 7, True, 0, True), (KB, 8, True, 0, False), (KB, 12, True, 0, False), (GAUSS, 5, True, 0, True), (GAUSS, 6, True, 0, False),
    (GAUSS, 8, True, 0, False), (KB, 8, False, 0, True), (GAUSS, 8, False, 0, True), (KB, 7, True, "FFT_2D", False),
    (KB, 7, True, "FFT_SPLIT", False)])
def test_second_buffer(lib, n, kernel, S, correct, flag, second):
    from paper_2504_00959_gb300 import _lib

    def size(flags):
        p = _lib.RickParams()
        assert lib.rick_params_default(ctypes.byref(p)) == 0
        p.n, p.nw, p.kernel, p.support = n, 16, kernel, S
        p.flags = 2 | (1 if correct else 0) | flags
        b = ctypes.c_size_t(0)
        assert lib.rick_workspace_size(ctypes.byref(p), 1000, ctypes.byref(b)) == 0
        return b.value
    more, buffer = size(getattr(_lib, flag) if flag else 0) - size(_lib.FFT_2D), 16 * 8 * n * n
    if second:
        assert buffer <= more <= 1.05 * buffer
    else:
        assert more == 0


@pytest.mark.parametrize("kernel", [GAUSS, KB])
@pytest.mark.parametrize("param", [1e-300, 1e-3, 700.0, 1e5, 1e300])
def test_extreme_kernel_parameters(lib, kernel, param):
    """A kernel parameter that no handle takes still gets an answer."""
    from paper_2504_00959_gb300 import _lib
    p = _lib.RickParams()
    assert lib.rick_params_default(ctypes.byref(p)) == 0
    p.n, p.nw, p.kernel, p.support, p.kernel_param = 1024, 4, kernel, 7, param
    b = ctypes.c_size_t(0)
    assert lib.rick_workspace_size(ctypes.byref(p), 1000, ctypes.byref(b)) == 0
    assert b.value >= 4 * 8 * 1024 * 1024
