"""Device memory that the graph replay of small problems costs: handles that replay share split
workspaces between steps the graph orders, and handles that never replay (batch members, the
grouped arithmetics of served solves) take no graph workspace and no staging copy."""
import ctypes
import random

import pytest

from helpers import build_host_probe

OWN, BATCH, SERVED = 0, 1, 2


@pytest.fixture(scope="module")
def probe():
    lib = build_host_probe("graph_memory_probe.cu", "graph_memory_probe")
    lib.probe_bytes.restype = lib.probe_group_partials.restype = ctypes.c_longlong
    return lib


def config(grid, o, v, precision=0, polish=0, **more):
    from paper_1911_00242_gb300 import binding
    return binding.make_config(grid, o, v, precision=precision, polish_precision=polish, diis_depth=6, **more)


# (grid, o, v, precision, MB of a handle whose steps use one workspace of two to four splits)
@pytest.mark.parametrize("grid,o,v,precision,mb", [((2, 2, 1), 6, 20, 0, 311.8), ((2, 2, 1), 8, 32, 0, 1512.6),
                                                   ((4, 1, 1), 4, 8, 0, 19.9), ((2, 2, 1), 7, 18, 0, 301.8),
                                                   ((2, 2, 2), 4, 16, 0, 675.1), ((3, 1, 1), 5, 13, 2, 103.8),
                                                   ((2, 2, 1), 6, 20, 1, 686.2)])
def test_footprint_of_small_handles(probe, grid, o, v, precision, mb):
    c = config(grid, o, v, precision)
    own, batch, served = (probe.probe_bytes(ctypes.byref(c), use) for use in (OWN, BATCH, SERVED))
    assert own < 1.5e6 * mb
    assert batch <= served <= own
    if precision != 2:
        assert batch == served


def test_replays_by_use(probe):
    """Bits 0..2: FP64, FP32 and double-float (Ozaki) arithmetics; 256: staging copy."""
    for precision, polish, own, served in ((0, 0, 1 + 256, 0), (1, 0, 3 + 256, 0), (1, 2, 7 + 256, 4), (2, 0, 5 + 256, 4)):
        c = config((3, 1, 1), 5, 13, precision, polish)
        assert probe.probe_replays(ctypes.byref(c), OWN) == own
        assert probe.probe_replays(ctypes.byref(c), BATCH) == 0
        assert probe.probe_replays(ctypes.byref(c), SERVED) == served
    big = config((2, 2, 2), 8, 32)
    assert probe.probe_replays(ctypes.byref(big), OWN) == 0


def test_steps_that_share_memory_are_ordered(probe):
    """Every pair of steps whose split partials or counters overlap is joined by a path of the
    graph's edges, over forms, layouts and sizes on both sides of the packed hole-hole rule."""
    rng = random.Random(11)
    sizes = [((2, 2, 2), 10, 5), ((2, 1, 1), 33, 6), ((1, 1, 1), 49, 10), ((2, 2, 1), 8, 32)]
    for _ in range(40):
        sizes.append((rng.choice([(1, 1, 1), (2, 1, 1), (3, 1, 1), (2, 2, 1), (3, 2, 1), (2, 2, 2)]),
                      rng.randint(1, 9), rng.randint(1, 24)))
    total = 0
    for grid, o, v in sizes:
        for precision, polish in ((0, 0), (1, 0), (1, 2), (2, 0)):
            for lean in (0, 1):
                c = config(grid, o, v, precision, polish, lean=lean)
                for use in (OWN, SERVED):
                    shared = ctypes.c_int(0)
                    bad = probe.probe_conflicts(ctypes.byref(c), use, ctypes.byref(shared))
                    assert bad == 0, (grid, o, v, precision, polish, lean, use)
                    total += shared.value
    assert total > 1000


def ranks(probe, c, dtype, fp32):
    out = []
    while True:
        order, own = (ctypes.c_int * 16)(), ctypes.c_int(-1)
        n = probe.probe_rank(ctypes.byref(c), dtype, fp32, len(out), order, ctypes.byref(own))
        if n < 0:
            return out
        out.append((own.value, list(order[:n])))


@pytest.mark.parametrize("grid,o,v", [((1, 1, 1), 6, 16), ((2, 1, 1), 4, 11), ((2, 2, 1), 8, 24), ((3, 1, 1), 5, 13)])
@pytest.mark.parametrize("fp32", [0, 1])
def test_autotuner_ranks_what_the_launch_reads(probe, grid, o, v, fp32):
    """For a group of one member the first candidate is the shape of the member's own plan (same
    model, same operand types, same splits), and mixed iterations, which read complex64 copies
    of complex128 integrals, rank as with integrals stored complex64."""
    c = config(grid, o, v, 1 if fp32 else 0)
    got = ranks(probe, c, 0, fp32)
    assert len(got) > 10
    for own, order in got:
        if order:
            assert sorted(order) == sorted(set(order))
            assert order[0] == own
    if fp32:
        assert got == ranks(probe, c, 1, fp32)


@pytest.mark.parametrize("fp32", [0, 1])
@pytest.mark.parametrize("members", [1, 4, 16, 64])
def test_grouped_split_partials_are_bounded(probe, fp32, members):
    """Beyond what its FP32 sums need, one grouped launch has at most 4 x 8 x 152 split items (twice
    the loads of half a mean CTA share), of at most 64 x 64 outputs."""
    for grid, o, v in (((2, 2, 1), 6, 20), ((2, 2, 2), 8, 24), ((1, 1, 1), 4, 8)):
        c = config(grid, o, v, 1 if fp32 else 0)
        gemm, got = 0, 0
        while got >= 0:
            for shape in range(12):
                least = ctypes.c_longlong(0)
                got = probe.probe_group_partials(ctypes.byref(c), members, fp32, gemm, shape, ctypes.byref(least))
                assert got <= 4 * 8 * 152 * 4096 + least.value, (grid, gemm, shape)
            gemm += 1
        assert gemm > 10


@pytest.mark.parametrize("count,seed,most", [(64, 2000, 26), (16, 4000, 13)])
@pytest.mark.parametrize("precision", [0, 1])
def test_served_solves_share_groups(probe, precision, count, seed, most):
    """Groups of the batched workload's 64 sizes and of the serving workload's 16, all served at
    once: no more than with a key of seven tile shapes picked by thresholds."""
    import ccsd_synth as cs
    keys = set()
    for s in cs.batch_specs(count, seed):
        c = config(s.grid, s.nocc, s.nvir, precision)
        out = (ctypes.c_longlong * 512)()
        n = probe.probe_key(ctypes.byref(c), precision, out, 512)
        assert 0 < n < 512
        keys.add(tuple(out[:n]))
    assert len(keys) <= most


@pytest.mark.parametrize("precision", [0, 1])
def test_served_launches_keep_k_groups(probe, precision):
    """Members of one group whose own shapes differ: each contraction launch has the K groups of all
    its members' own shapes, so their sums keep their order."""
    split = 0
    for one, two in ((((2, 2, 1), 4, 8), ((2, 2, 1), 6, 14)), (((3, 1, 1), 2, 5), ((3, 1, 1), 7, 20)),
                     (((3, 1, 1), 3, 7), ((3, 1, 1), 8, 13)), (((2, 2, 1), 5, 18), ((2, 2, 1), 8, 20))):
        a, b = (config(*x, precision) for x in (one, two))
        gemm = 0
        while True:
            n = probe.probe_classes(ctypes.byref(a), ctypes.byref(b), precision, gemm)
            if n < 0:
                break
            assert n < 4
            split += n > 1
            gemm += 1
        assert gemm > 10
    assert split > 0
