"""Small problems replay the residual as a CUDA graph built from the plan's data
dependencies.  The replayed kernels are those of the step-by-step path (which tracing
takes), so the residual and the iterates must be equal to it bit for bit, for every form,
operand layout and integral type, also with a handle per stream running side by side."""
import numpy as np
import pytest

import ccsd_synth as cs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FORMS = [dict(precision=0), dict(precision=1), dict(precision=2), dict(precision=1, polish_precision=2)]


def problem(grid, o, v, dtype):
    spec = cs.SynthSpec(grid, o, v, 5200 + o + v, time_reversal=False, fock_offdiag=0.02, int_dtype=dtype)
    dev = {k: torch.from_numpy(np.ascontiguousarray(x)).cuda() for k, x in cs.generate(spec).items()}
    t = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in cs.random_amplitudes(spec, 5, 0.02)]
    return dev, t


def outputs(S, t, n, precision):
    S.set_precision(precision)
    r = [torch.empty_like(x) for x in t]
    S.residual(*t, *r)
    S.set_amplitudes(*t)
    S.iterate(n)
    a = [torch.empty_like(x) for x in t]
    S.get_amplitudes(*a)
    torch.cuda.synchronize()
    return r + a


@pytest.mark.parametrize("lean", [0, 1])
@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("grid,o,v,dtype", [((1, 1, 1), 2, 19, "c128"), ((2, 1, 1), 3, 9, "c64"),
                                            ((3, 1, 1), 4, 7, "c128"), ((2, 2, 1), 5, 12, "c64")])
def test_replay_equals_step_by_step(lib, grid, o, v, dtype, form, lean):
    from paper_1911_00242_gb300.binding import Solver
    dev, t = problem(grid, o, v, dtype)
    S = Solver(grid, o, v, dev, diis_depth=4, lean=lean, conv_tol=0.0, **form)
    for precision in sorted({0, form["precision"], form.get("polish_precision", 0)}):
        S.trace(True)
        want = outputs(S, t, 3, precision)
        S.trace(False)
        for _ in range(3):
            for x, y in zip(outputs(S, t, 3, precision), want):
                assert torch.equal(x, y)
    S.close()


def test_handles_on_their_own_streams(lib):
    """Four handles of two sizes, each on its own stream, with their residuals in flight
    together: each gives what it gives alone."""
    from paper_1911_00242_gb300.binding import Solver
    sizes = [((2, 1, 1), 3, 9), ((3, 1, 1), 4, 7), ((2, 1, 1), 3, 9), ((3, 1, 1), 4, 7)]
    streams = [torch.cuda.Stream() for _ in sizes]
    S, T, R, want = [], [], [], []
    for (grid, o, v), st in zip(sizes, streams):
        dev, t = problem(grid, o, v, "c128")
        torch.cuda.synchronize()
        s = Solver(grid, o, v, dev, stream=st.cuda_stream)
        r = [torch.empty_like(x) for x in t]
        s.trace(True)
        s.residual(*t, *r)
        torch.cuda.synchronize()
        want.append([x.clone() for x in r])
        s.trace(False)
        S.append(s), T.append(t), R.append(r)
    for _ in range(20):
        for s, t, r in zip(S, T, R):
            s.residual(*t, *r)
    torch.cuda.synchronize()
    for r, w in zip(R, want):
        assert all(torch.equal(x, y) for x, y in zip(r, w))
    for s in S:
        s.close()


def test_residual_inside_a_callers_capture(lib):
    """A caller may capture the FP64 residual into a graph of its own (no host
    synchronization in it): the launches join that capture."""
    from paper_1911_00242_gb300.binding import Solver
    dev, t = problem((2, 1, 1), 3, 9, "c128")
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    S = Solver((2, 1, 1), 3, 9, dev, stream=st.cuda_stream)
    r = [torch.empty_like(x) for x in t]
    S.residual(*t, *r)
    torch.cuda.synchronize()
    want = [x.clone() for x in r]
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        S.residual(*t, *r)
    for x in r:
        x.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert all(torch.equal(x, y) for x, y in zip(r, want))
    S.close()
