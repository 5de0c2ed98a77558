"""Served solves of uneven sizes that share groups although their own plans take different tile
shapes, K groups and splits: each must end with the energy it has alone, bit for bit."""
import time

import pytest

import ccsd_synth as cs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SPECS = [cs.SynthSpec((2, 1, 1), 1, 4, 3301), cs.SynthSpec((2, 1, 1), 3, 17, 3302), cs.SynthSpec((2, 1, 1), 7, 9, 3303),
         cs.SynthSpec((3, 1, 1), 3, 7, 3304), cs.SynthSpec((3, 1, 1), 8, 13, 3305),
         cs.SynthSpec((1, 1, 1), 4, 30, 3306, time_reversal=False)]


def serve(jobs):
    from paper_1911_00242_gb300.binding import Server
    srv = Server(64 << 30, 16)
    ids = [srv.submit(s.grid, s.nocc, s.nvir, inp, **cfg) for s, inp, cfg in jobs]
    done, t0 = {}, time.time()
    while len(done) < len(ids):
        for i in ids:
            st, e, t, it = srv.poll(i)
            if st == 2 or st < 0:
                done[i] = (st, e)
        assert time.time() - t0 < 300.0, "serving loop did not finish"
        time.sleep(0.005)
    srv.close()
    return [done[i] for i in ids]


def alone(job):
    from paper_1911_00242_gb300.binding import Solver
    s, inp, cfg = job
    S = Solver(s.grid, s.nocc, s.nvir, inp, **cfg)
    S.solve()
    e = S.energy().real
    S.close()
    return e


@pytest.mark.parametrize("precision,polish", [(0, 0), (1, 0), (1, 2)])
def test_uneven_sizes_in_one_mix(lib, precision, polish):
    cfg = dict(conv_tol=1e-8, diis_depth=6, max_iter=100, precision=precision, polish_precision=polish, mixed_tol=1e-7,
               polish_iters=3)
    jobs = [(s, cs.generate(s), cfg) for s in SPECS]
    for job, (st, e) in zip(jobs, serve(jobs)):
        assert st == 2, job[0]
        assert e == alone(job), job[0]


def test_diis_depths_in_one_mix(lib):
    """Requests that differ in their DIIS depth only."""
    inp = cs.generate(SPECS[0])
    jobs = [(SPECS[0], inp, dict(conv_tol=1e-8, diis_depth=d, max_iter=200)) for d in (0, 4, 6)]
    for job, (st, e) in zip(jobs, serve(jobs)):
        assert st == 2, job[2]
        assert e == alone(job), job[2]
