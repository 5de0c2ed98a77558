"""The first residual of a handle, which builds its graph, while the same thread captures another
stream: the capture must go on and the residual must be the one the handle gives alone."""
import numpy as np
import pytest

import ccsd_synth as cs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["thread_local", "global"])
def test_first_residual_beside_a_capture(lib, mode):
    from paper_1911_00242_gb300.binding import Solver
    grid, o, v = (2, 1, 1), 3, 9
    spec = cs.SynthSpec(grid, o, v, 5400, time_reversal=False, fock_offdiag=0.02)
    dev = {k: torch.from_numpy(np.ascontiguousarray(x)).cuda() for k, x in cs.generate(spec).items()}
    t = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in cs.random_amplitudes(spec, 5, 0.02)]
    r = [torch.empty_like(x) for x in t]
    own, other = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    alone = Solver(grid, o, v, dev, stream=own.cuda_stream)
    alone.residual(*t, *r)
    torch.cuda.synchronize()
    want = [x.clone() for x in r]
    for x in r:
        x.zero_()
    count = torch.zeros(1024, device="cuda")
    S = Solver(grid, o, v, dev, stream=own.cuda_stream)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=other, capture_error_mode=mode):
        count += 1
        S.residual(*t, *r)
        count += 1
    g.replay()
    torch.cuda.synchronize()
    assert bool((count == 2).all())
    assert all(torch.equal(x, y) for x, y in zip(r, want))
    S.close()
    alone.close()
