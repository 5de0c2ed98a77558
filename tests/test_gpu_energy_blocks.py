"""ccsd_energy at block lengths (o v)^2 on both sides of the rule that sums short blocks flat, and of
its 2048-element units: against numpy in complex128.  The bar is 1e-14 of the sum of the terms'
moduli: each partial sum has at most a few hundred terms per thread, added in a tree."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.complex128, torch.complex64])
@pytest.mark.parametrize("grid,o,v", [((1, 1, 1), 1, 1), ((1, 1, 1), 1, 45), ((3, 1, 1), 1, 2), ((3, 3, 3), 2, 6), ((5, 1, 1), 3, 15),
                                      ((3, 2, 1), 2, 21), ((2, 2, 2), 4, 16), ((3, 1, 1), 5, 23), ((2, 2, 1), 9, 13)])
def test_energy(lib, grid, o, v, dtype):
    from paper_1911_00242_gb300.binding import Solver
    N, dim = math.prod(grid), {"o": o, "v": v}
    gen = torch.Generator(device="cuda").manual_seed(100 * o + v)

    def rand(*shape):
        return torch.randn(shape, dtype=torch.complex128, device="cuda", generator=gen)

    a = {b: (0.01 * rand(N, N, N, *(dim[x] for x in b))).to(dtype) for b in ("oooo", "ooov", "oovv", "ovvo", "ovvv", "vvvv")}
    for name, p, q, e in (("f_oo", o, o, -1.0), ("f_vv", v, v, 1.0), ("f_ov", o, v, None)):
        a[name] = 0.01 * rand(N, p, q)
        if e is not None:
            a[name].diagonal(dim1=1, dim2=2).fill_(e)
    t1, t2 = rand(N, o, v), rand(N, N, N, o, o, v, v)
    S = Solver(grid, o, v, a)
    S.set_amplitudes(t1, t2)
    got = S.energy()
    S.close()
    t1, t2, f = (x.cpu().numpy() for x in (t1, t2, a["f_ov"]))
    g = a["oovv"].cpu().numpy().astype(np.complex128)
    terms = [f * t1, 0.25 * g * t2]
    for i in range(N):                       # 1/2 <i ki j kj||a ki b kj> t_i^a t_j^b
        terms.append(0.5 * g[i, :, i] * t1[i][None, :, None, :, None] * t1[:, None, :, None, :])
    want = sum(x.sum() for x in terms) / N
    size = sum(np.abs(x).sum() for x in terms) / N
    assert abs(got - want) < 1e-14 * size
