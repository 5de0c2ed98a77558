"""Graph replays of plans with the packed tensor-core hole-hole contractions, where the ladder reads
the tau operand that an earlier step embedded and a contraction is up to four mirrored launches:
equal to the step-by-step path bit for bit.  A batch's captured iteration, whose steps run side
by side, gives the same bits every time it is replayed from the same amplitudes."""
import numpy as np
import pytest

import ccsd_synth as cs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def problem(grid, o, v, dtype="c128"):
    spec = cs.SynthSpec(grid, o, v, 5500 + o + v, time_reversal=False, fock_offdiag=0.02, int_dtype=dtype)
    dev = {k: torch.from_numpy(np.ascontiguousarray(x)).cuda() for k, x in cs.generate(spec).items()}
    t = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in cs.random_amplitudes(spec, 5, 0.02)]
    return dev, t


@pytest.mark.parametrize("form", [dict(precision=1, polish_precision=2), dict(precision=2)])
@pytest.mark.parametrize("grid,o,v,dtype", [((2, 2, 2), 10, 5, "c128"), ((2, 1, 1), 33, 6, "c64"), ((1, 1, 1), 49, 10, "c128")])
def test_packed_replay_equals_step_by_step(lib, grid, o, v, dtype, form):
    from paper_1911_00242_gb300.binding import Solver
    assert 8.0 * (grid[0] * grid[1] * grid[2]) ** 4 * o ** 4 * v ** 2 >= 4e9
    dev, t = problem(grid, o, v, dtype)
    S = Solver(grid, o, v, dev, **form)
    for precision in sorted({form["precision"], form.get("polish_precision", form["precision"])}):
        S.set_precision(precision)
        got = []
        for trace in (True, False, False, False):
            S.trace(trace)
            r = [torch.full_like(x, float("nan")) for x in t]
            S.residual(*t, *r)
            torch.cuda.synchronize()
            got.append(r)
        for r in got[1:]:
            assert all(torch.equal(x, y) for x, y in zip(r, got[0])), precision
    S.close()


@pytest.mark.parametrize("grid,o,v,dtype", [((2, 2, 2), 14, 5, "c128"), ((2, 1, 1), 45, 6, "c64"), ((3, 1, 1), 40, 8, "c64"),
                                            ((1, 1, 1), 49, 20, "c128")])
def test_packed_mixed_residual(lib, grid, o, v, dtype):
    """The mixed form from its own line on, against the FP64 form, replayed and step by step (bar as
    for the parity tests: 1e-5 of max|R|)."""
    from paper_1911_00242_gb300.binding import Solver
    assert 8.0 * (grid[0] * grid[1] * grid[2]) ** 4 * o ** 4 * v ** 2 >= (6e10 if grid[0] == 3 else 1.6e10)
    dev, t = problem(grid, o, v, dtype)
    got = []
    for precision in (0, 1):
        S = Solver(grid, o, v, dev, precision=precision)
        for trace in (False, True):
            S.trace(trace)
            r = [torch.full_like(x, float("nan")) for x in t]
            S.residual(*t, *r)
            torch.cuda.synchronize()
            got.append(r)
        S.close()
    top = max(float(x.abs().max()) for x in got[0])
    for x, y, z in zip(got[0], got[2], got[3]):
        assert torch.equal(y, z)
        assert float((x - y).abs().max()) < 1e-5 * top


@pytest.mark.parametrize("precision", [0, 1])
def test_batch_replays_agree(lib, precision):
    """Members on both sides of the packing rule (mixed), of uneven sizes, with DIIS."""
    import ctypes
    from paper_1911_00242_gb300 import binding
    sizes = [((2, 2, 2), 14, 5), ((2, 1, 1), 3, 9), ((2, 2, 1), 5, 12), ((2, 1, 1), 45, 6), ((3, 1, 1), 4, 7)]
    probs = [problem(*s) for s in sizes]
    B = binding.BatchSolver([(g, o, v, d) for (g, o, v), (d, _) in zip(sizes, probs)], precision=precision, diis_depth=4,
                            conv_tol=0.0)
    B.iterate(1)
    got = []
    for _ in range(4):
        for i, (_, t) in enumerate(probs):
            h = ctypes.c_void_p()
            binding.check(lib.ccsd_batch_member(B.h, i, ctypes.byref(h)), "ccsd_batch_member")
            binding.check(lib.ccsd_set_amplitudes(h, t[0].data_ptr(), t[1].data_ptr()), "ccsd_set_amplitudes")
        B.iterate(3)
        out = []
        for i, (_, t) in enumerate(probs):
            a = [torch.empty_like(x) for x in t]
            B.member_amplitudes(i, *a)
            out += a
        torch.cuda.synchronize()
        got.append(out)
    for out in got[1:]:
        assert all(torch.equal(x, y) for x, y in zip(out, got[0]))
    B.close()
