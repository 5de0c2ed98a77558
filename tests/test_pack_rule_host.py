"""Where the tensor-core hole-hole contractions are packed by antisymmetry: from 4e9 flops on in the
Ozaki arithmetic and, in the mixed one, from 4e9, 1.6e10 or 6e10 on by the number of pair classes
of the grid (below, a residual was slower packed); each set by its own line in a handle that has
both, and never in the lean layout."""
import pytest


def packed(grid, o, v, **more):
    """Whether the tensor-core hole_hole GEMMs of the mixed set (mode 2) and the Ozaki set (mode 5)
    run a fraction of the full sum's flops; None where the handle has no such set."""
    from paper_1911_00242_gb300 import binding
    n = {}
    for name, kind, mode, flops in binding.plan_describe(grid, o, v, **more):
        if kind == 6 and name == "hole_hole":
            n[mode] = n.get(mode, 0.0) + flops
    full = 8.0 * (grid[0] * grid[1] * grid[2]) ** 4 * o ** 4 * v ** 2
    return tuple(n[m] < 0.6 * full if m in n else None for m in (2, 5))


@pytest.mark.parametrize("grid,o,v,line", [((1, 1, 1), 32, 22, 4e9), ((1, 1, 1), 32, 24, 4e9),
                                           ((2, 2, 1), 8, 32, 1.6e10), ((2, 2, 2), 8, 10, 1.6e10), ((2, 2, 2), 8, 12, 1.6e10),
                                           ((3, 1, 1), 16, 12, 6e10), ((4, 1, 1), 10, 30, 6e10), ((3, 2, 1), 8, 28, 6e10),
                                           ((3, 1, 1), 20, 26, 6e10)])
def test_lines(grid, o, v, line):
    n = 8.0 * (grid[0] * grid[1] * grid[2]) ** 4 * o ** 4 * v ** 2
    assert packed(grid, o, v, precision=1) == (n >= line, None)
    assert packed(grid, o, v, precision=2) == (None, n >= 4e9)
    assert packed(grid, o, v, precision=1, polish_precision=2) == (n >= line, n >= 4e9)
    assert packed(grid, o, v, precision=1, polish_precision=2, lean=1) == (False, False)
