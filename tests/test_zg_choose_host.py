"""The SIMT GEMM's choice of K splits, from one output to the output counts of 27 k points:
at least the splits that bound an FP32 partial sum, at most one split per 32 terms, and no
more than 2^26 partials a launch unless the FP32 bound needs them."""
import ctypes

import pytest

from helpers import build_host_probe


@pytest.fixture(scope="module")
def probe():
    lib = build_host_probe("zg_choose_probe.cu", "zg_choose_probe")
    lib.probe_zg_choose.argtypes = [ctypes.c_int] * 4 + [ctypes.c_longlong] * 2 + [ctypes.POINTER(ctypes.c_int)]
    lib.probe_zg_least.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_longlong]
    lib.probe_zg_least.restype = ctypes.c_longlong
    return lib


@pytest.mark.parametrize("arith", [0, 1, 2])
def test_splits_are_bounded(probe, arith):
    shape = ctypes.c_int(0)
    for M, N in ((1, 1), (8, 8), (65, 65), (576, 64), (1024, 64), (4096, 1024)):
        for K in (1, 8, 33, 192, 4096):
            for nchunk in (1, 27, 729):
                for nbatch in (1, 8, 729, 19683):
                    ns = probe.probe_zg_choose(arith, M, N, K, nchunk, nbatch, ctypes.byref(shape))
                    least = probe.probe_zg_least(arith, K, nchunk)
                    units = nchunk * ((K + 31) // 32)
                    assert 0 <= shape.value < 12
                    assert least <= ns <= max(least, units)
                    assert ns == least or ns * nbatch * M * N <= 1 << 26
