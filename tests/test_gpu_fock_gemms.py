"""Fock-like terms of Ozaki iterations on both sides of the amplitude count that splits them
(GEMMs on double-float copies above, one fused pass below), against the FP64 form of the same
problem; odd orbital counts, off the tile widths.  Bar as for the parity tests: 1e-11 of max|R|."""
import numpy as np
import pytest

import ccsd_synth as cs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid,o,v,gemms,dtype", [((2, 1, 1), 27, 27, True, "c128"), ((3, 1, 1), 20, 21, True, "c64"),
                                                  ((3, 1, 1), 19, 20, False, "c128"), ((1, 1, 1), 45, 47, True, "c128")])
def test_fock_terms_at_the_line(lib, grid, o, v, gemms, dtype):
    from paper_1911_00242_gb300.binding import CCSD_FP64, CCSD_OZAKI, Solver
    n = grid[0] * grid[1] * grid[2]
    assert (n ** 3 * o ** 2 * v ** 2 >= 1 << 22) == gemms
    spec = cs.SynthSpec(grid, o, v, 7300 + o + v, time_reversal=False, fock_offdiag=0.02, int_dtype=dtype)
    dev = {k: torch.from_numpy(np.ascontiguousarray(x)).cuda() for k, x in cs.generate(spec).items()}
    t = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in cs.random_amplitudes(spec, 6, 0.02)]
    out = []
    for precision in (CCSD_FP64, CCSD_OZAKI):
        S = Solver(grid, o, v, dev, precision=precision)
        r = [torch.empty_like(x) for x in t]
        S.residual(*t, *r)
        torch.cuda.synchronize()
        S.close()
        out.append(r)
    top = max(float(x.abs().max()) for x in out[0])
    for x, y in zip(*out):
        assert float((x - y).abs().max()) < 1e-11 * top
