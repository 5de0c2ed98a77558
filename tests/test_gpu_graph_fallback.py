"""A residual graph that cannot be instantiated is no error: the handle launches its steps one
by one, with the same bits.  The failing call is a fake (an error code from a wrapped
cudaGraphInstantiate in a second link of the library's objects); nothing faults on the device."""
import numpy as np
import pytest

import ccsd_synth as cs
from helpers import load_with_fakes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wrapped(lib):
    """The library with a fake in place of cudaGraphInstantiate."""
    from paper_1911_00242_gb300 import binding
    save = binding._lib
    binding._lib = load_with_fakes("graph_fallback_wrap.cpp", ["cudaGraphInstantiate"])
    try:
        yield binding._lib
    finally:
        binding._lib = save


@pytest.mark.parametrize("precision", [0, 1, 2])
def test_failed_instantiation_falls_back(wrapped, precision):
    from paper_1911_00242_gb300.binding import Solver
    grid, o, v = (2, 1, 1), 3, 9
    spec = cs.SynthSpec(grid, o, v, 5300, time_reversal=False, fock_offdiag=0.02)
    dev = {k: torch.from_numpy(np.ascontiguousarray(x)).cuda() for k, x in cs.generate(spec).items()}
    t = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in cs.random_amplitudes(spec, 5, 0.02)]
    got = []
    for fail in (0, 1):
        calls = wrapped.probe_instantiate_calls()
        S = Solver(grid, o, v, dev, precision=precision, diis_depth=4, conv_tol=0.0)
        wrapped.probe_fail_instantiate(fail)
        try:
            r, a = ([torch.full_like(x, float("nan")) for x in t] for _ in range(2))
            S.residual(*t, *r)
            S.set_amplitudes(*t)
            S.iterate(3)
            S.get_amplitudes(*a)
            torch.cuda.synchronize()
            assert wrapped.ccsd_last_error() == b""
        finally:
            wrapped.probe_fail_instantiate(0)
        S.close()
        # both graphs are built, or the first failure is the last try
        assert wrapped.probe_instantiate_calls() - calls == (1 if fail else 2)
        got.append(r + a)
    assert all(torch.equal(x, y) for x, y in zip(*got))
