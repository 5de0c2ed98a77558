"""f64_scaled (the tensor-core epilogues' float-to-double widening by integer operations)
against numpy's exact conversion and scaling, bit for bit: normal floats at both ends of
the range, subnormals, signed zeros, infinities and NaN, and exponents up to the largest
the epilogues use (two row scales of 2^120 and alpha)."""
import ctypes

import numpy as np
import pytest

from helpers import build_host_probe


@pytest.fixture(scope="module")
def probe():
    lib = build_host_probe("f64_scaled_probe.cu", "f64_scaled_probe")
    lib.probe_f64_scaled.argtypes = [ctypes.c_void_p, ctypes.c_longlong, ctypes.c_int, ctypes.c_int, ctypes.c_void_p]
    lib.probe_pow2.argtypes = [ctypes.c_double, ctypes.POINTER(ctypes.c_int)]
    return lib


@pytest.mark.parametrize("e", [0, -1, 1, 17, -120, 240, -242])
@pytest.mark.parametrize("neg", [0, 1])
def test_widening_is_exact(probe, e, neg):
    rng = np.random.default_rng(3)
    bits = rng.integers(0, 2 ** 32, 20000, dtype=np.uint64).astype(np.uint32)
    edge = np.array([0, 1, 0x007fffff, 0x00800000, 0x00800001, 0x3f800000, 0x7f7fffff, 0x7f800000, 0x7fc00000],
                    np.uint32)
    x = np.concatenate([bits, edge, edge | np.uint32(0x80000000)]).view(np.float32)
    out = np.empty(x.size)
    probe.probe_f64_scaled(x.ctypes.data, x.size, e, neg, out.ctypes.data)
    with np.errstate(invalid="ignore"):        # signalling NaN patterns
        want = np.ldexp((-x if neg else x).astype(np.float64), e)
    nan = np.isnan(want)
    assert np.array_equal(np.isnan(out), nan)
    assert np.array_equal(out[~nan].view(np.uint64), want[~nan].view(np.uint64))


def test_powers_of_two(probe):
    e = ctypes.c_int(0)
    for k in (-200, -1, 0, 1, 200):
        assert probe.probe_pow2(2.0 ** k, ctypes.byref(e)) == 1 and e.value == k
    for p in (0.0, 3.0, 0.75, 2.0 ** 201, 2.0 ** -201, float("inf"), float("nan"), 5e-324):
        assert probe.probe_pow2(p, ctypes.byref(e)) == 0, p
