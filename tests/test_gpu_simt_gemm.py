"""The SIMT complex GEMM's tile shapes and K splits, against the oracle's residual.

Sizes at which they can go wrong: contractions of one chunk whose K is split (N_k = 1
with a long K), K and outputs one above and one below the 8-, 16- and 32-wide tiles,
single rows and columns, and blocks that leave whole warps of a tile empty.  Every
residual is evaluated twice on one handle: the split tiles' counters must return to
zero.  Bars as for the parity tests: FP64 1e-12 absolute, elementwise (sums of at most
1e5 terms of size at most 1e-2 in another order); Ozaki 1e-11 and mixed 1e-5 of
max|R|."""
import numpy as np
import pytest

import ccsd_synth as cs
from oracle import ccsd_k

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES = [((1, 1, 1), 2, 33), ((1, 1, 1), 1, 17), ((1, 1, 1), 9, 15), ((2, 1, 1), 8, 9), ((2, 1, 1), 3, 31),
          ((3, 1, 1), 5, 13), ((1, 1, 1), 17, 7), ((2, 1, 1), 1, 1)]


@pytest.mark.parametrize("grid,o,v", SHAPES)
@pytest.mark.parametrize("dtype", ["c128", "c64"])
def test_residual_at_tile_edges(lib, grid, o, v, dtype):
    from paper_1911_00242_gb300.binding import CCSD_FP64, CCSD_MIXED, CCSD_OZAKI, Solver
    spec = cs.SynthSpec(grid, o, v, 4100 + 10 * o + v, time_reversal=False, fock_offdiag=0.02, int_dtype=dtype)
    inp = cs.generate(spec)
    t1, t2 = cs.random_amplitudes(spec, 7)
    P = ccsd_k.Problem(grid, o, v, {k: np.asarray(x, np.complex128) for k, x in inp.items()})
    q1, q2 = ccsd_k.residual(P, t1, t2)
    top = max(np.abs(q1).max(), np.abs(q2).max())
    dev = {k: torch.from_numpy(np.ascontiguousarray(x)).cuda() for k, x in inp.items()}
    a1, a2 = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (t1, t2))
    for precision, bar in ((CCSD_FP64, 1e-12), (CCSD_OZAKI, 1e-11 * top), (CCSD_MIXED, 1e-5 * top)):
        S = Solver(grid, o, v, dev, precision=precision)
        r1, r2 = torch.empty_like(a1), torch.empty_like(a2)
        for _ in range(2):
            r1.fill_(float("nan"))
            r2.fill_(float("nan"))
            S.residual(a1, a2, r1, r2)
            torch.cuda.synchronize()
            assert np.abs(r1.cpu().numpy() - q1).max() < bar, precision
            assert np.abs(r2.cpu().numpy() - q2).max() < bar, precision
        S.close()
