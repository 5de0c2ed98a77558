"""The antisymmetry-packed tensor-core hole-hole contractions against the FP64 form of the
same handle's problem, at sizes that take them: grids with and without classes of unequal
momenta, odd orbital counts, pair lists off
the tile widths.  Bars as for the parity tests: Ozaki 1e-11, mixed 1e-5 of max|R|."""
import numpy as np
import pytest

import ccsd_synth as cs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid,o,v,dtype", [((2, 2, 2), 10, 5, "c128"), ((3, 2, 1), 13, 6, "c64"), ((1, 1, 1), 49, 10, "c128"),
                                            ((2, 1, 1), 33, 6, "c128")])
def test_packed_hole_hole(lib, grid, o, v, dtype):
    from paper_1911_00242_gb300.binding import CCSD_FP64, CCSD_MIXED, CCSD_OZAKI, Solver
    n = grid[0] * grid[1] * grid[2]
    assert 8.0 * n ** 4 * o ** 4 * v ** 2 >= 4e9
    spec = cs.SynthSpec(grid, o, v, 6100 + o + v, time_reversal=False, fock_offdiag=0.02, int_dtype=dtype)
    dev = {k: torch.from_numpy(np.ascontiguousarray(x)).cuda() for k, x in cs.generate(spec).items()}
    t = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in cs.random_amplitudes(spec, 5, 0.02)]
    want = None
    for precision, bar in ((CCSD_FP64, 0.0), (CCSD_OZAKI, 1e-11), (CCSD_MIXED, 1e-5)):
        S = Solver(grid, o, v, dev, precision=precision)
        r = [torch.empty_like(x) for x in t]
        S.residual(*t, *r)
        torch.cuda.synchronize()
        S.close()
        if want is None:
            want = r
            top = max(float(x.abs().max()) for x in r)
            continue
        for x, y in zip(r, want):
            assert float((x - y).abs().max()) < bar * top, precision
