"""The autotuner of a batch when device memory for split partials cannot be had: candidates that
need it are skipped, and the launch that stays runs without.  The failing call is a fake (an
error code from a wrapped cudaMalloc in a second link of the library's objects)."""
import numpy as np
import pytest

import ccsd_synth as cs
from helpers import load_with_fakes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wrapped(lib):
    from paper_1911_00242_gb300 import binding
    save = binding._lib
    binding._lib = load_with_fakes("batch_alloc_wrap.cpp", ["cudaMalloc"])
    try:
        yield binding._lib
    finally:
        binding._lib = save


def test_tuning_without_room_for_splits(wrapped):
    """Energies as with room: the sums are added in another order (bar of the batch tests)."""
    from paper_1911_00242_gb300.binding import BatchSolver
    specs = [cs.SynthSpec((2, 2, 1), 6, 20, 2106 + i) for i in range(2)]
    devs = [{k: torch.from_numpy(np.ascontiguousarray(x)).cuda() for k, x in cs.generate(s).items()} for s in specs]
    got, refused = [], []
    for limit in (0, 1 << 14):
        B = BatchSolver([(s.grid, s.nocc, s.nvir, d) for s, d in zip(specs, devs)], conv_tol=0.0)
        wrapped.probe_limit_alloc(limit)
        try:
            B.iterate(3)                       # the first iteration tunes
            refused.append(wrapped.probe_refused())
        finally:
            wrapped.probe_limit_alloc(0)
        got.append(B.energies())
        B.close()
    assert refused[0] == 0 and refused[1] > 0
    assert max(abs(x - y) for x, y in zip(*got)) < 1e-12
