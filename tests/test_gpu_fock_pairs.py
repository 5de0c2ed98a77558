"""Ozaki iterations' fused Fock-like terms (two elements i, i + 1 a thread) and ladder W' rows
against the FP64 form of the same problem: one, two and odd numbers of occupied orbitals,
virtual counts off the warp width, both integral types.  Bar as for the parity tests: 1e-11
of max|R|."""
import numpy as np
import pytest

import ccsd_synth as cs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid,o,v,dtype", [((3, 1, 1), 1, 5, "c128"), ((2, 2, 1), 2, 7, "c64"), ((3, 1, 1), 3, 12, "c64"),
                                            ((2, 1, 1), 7, 33, "c128"), ((1, 1, 1), 9, 31, "c128")])
def test_fused_fock_and_ladder_w(lib, grid, o, v, dtype):
    from paper_1911_00242_gb300.binding import CCSD_FP64, CCSD_OZAKI, Solver
    spec = cs.SynthSpec(grid, o, v, 8200 + o + v, time_reversal=False, fock_offdiag=0.02, int_dtype=dtype)
    dev = {k: torch.from_numpy(np.ascontiguousarray(x)).cuda() for k, x in cs.generate(spec).items()}
    t = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in cs.random_amplitudes(spec, 7, 0.05)]
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
