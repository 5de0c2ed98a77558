"""The work that users of the library time: residuals, iterations, solves, batches and
energies of periodic CCSD problems, through the Python binding.

A case is one problem: the k grid (n1, n2, n3), occupied / virtual spin orbitals per k,
the arithmetic (fp64, ozaki, mixed), the element type of the integrals, and what is
called.  Inputs are drawn on the GPU with the symmetries of antisymmetrized integrals:
each Bloch-normalized <pq||rs> has standard deviation 0.05 / N_k, occupied levels lie in
[-1.5, -0.5] Ha and virtual ones in [0.5, 2.5] Ha; with time reversal
x(-k) = conj(x(k)); `fock` is the size of an off-diagonal Fock matrix (0: canonical).
"""
import ctypes
import math

import numpy as np
import torch

from paper_1911_00242_gb300 import binding

PRECISION = {"fp64": binding.CCSD_FP64, "ozaki": binding.CCSD_OZAKI, "mixed": binding.CCSD_MIXED}
BLOCKS = ("oooo", "ooov", "oovv", "ovvo", "ovvv", "vvvv")
DIIS = 6
# grids of up to 8 k points: molecule-like cells, chains, slabs and small 3D meshes
GRIDS = ((1, 1, 1), (2, 1, 1), (3, 1, 1), (2, 2, 1), (4, 1, 1), (5, 1, 1), (3, 2, 1), (2, 2, 2))
SOLVE_TOL = 1e-12
SOLVE_ITERATIONS = 30           # updates a solve to SOLVE_TOL takes, about, for work()


def case(name, call, grid, o, v, form, ints="c128", fock=0.0, time_reversal=True, **more):
    return dict(name=name, call=call, n1=grid[0], n2=grid[1], n3=grid[2], o=o, v=v, form=form, ints=ints, fock=fock,
                time_reversal=time_reversal, **more)


def listed():
    return [
        # one residual of a short chain, the smallest problem of the test suite's workloads:
        # an outer loop (a geometry scan, a Newton solver) calls this many times
        case("fp64_residual_chain", "residual", (4, 1, 1), 4, 8, "fp64"),
        # iterations with DIIS of an odd-sized, non-canonical, complex problem in FP64
        case("fp64_iterate_odd", "iterate", (3, 1, 1), 5, 13, "fp64", ints="c64", fock=0.02, time_reversal=False,
             updates=3),
        # the benchmark's workload: one FP64 iteration of the 2x2x2 grid
        case("fp64_iterate_grid222", "iterate", (2, 2, 2), 8, 32, "fp64", updates=1),
        # the same workload's residual with FP64 accuracy from the tensor cores
        case("ozaki_residual_grid222", "residual", (2, 2, 2), 8, 32, "ozaki"),
        # iterations with DIIS of the 2x2x1 slab, integrals stored complex64
        case("ozaki_iterate_grid221", "iterate", (2, 2, 1), 8, 32, "ozaki", ints="c64", updates=2),
        # a small odd problem, for which every launch is short
        case("ozaki_residual_odd", "residual", (3, 1, 1), 5, 13, "ozaki", fock=0.02, time_reversal=False),
        # whole solves from t = 0: mixed iterations, then polish iterations to a tight
        # threshold (as properties and gradients need it)
        case("mixed_solve_grid222", "solve", (2, 2, 2), 6, 24, "mixed", polish="ozaki"),
        case("mixed_solve_grid221", "solve", (2, 2, 1), 6, 20, "mixed", ints="c64", polish="fp64"),
        case("mixed_solve_chain", "solve", (4, 1, 1), 4, 8, "mixed", polish="ozaki"),
        # twelve independent problems of uneven size, advanced together
        case("fp64_batch", "batch", (1, 1, 1), 6, 16, "fp64", members=12, updates=1),
        # the energy of held amplitudes, after every iteration of a user's own loop
        case("energy_grid222", "energy", (2, 2, 2), 8, 32, "fp64"),
    ]


def draw(rng):
    call = rng.choice(("residual", "residual", "iterate", "iterate", "solve", "batch", "energy"))
    form = {"residual": ("fp64", "ozaki", "ozaki"), "iterate": ("fp64", "ozaki", "ozaki"), "solve": ("mixed",),
            "batch": ("fp64",), "energy": ("fp64",)}[call]
    form = rng.choice(form)
    grid = rng.choice(GRIDS)
    o = rng.randint(2, 8)
    v = int(round(math.exp(rng.uniform(math.log(6), math.log(32)))))
    c = case("", call, grid, o, v, form, ints=rng.choice(("c128", "c64")), fock=rng.choice((0.0, 0.02)),
             time_reversal=rng.random() < 0.7)
    del c["name"]
    if call == "iterate":
        c["updates"] = 1 if flops(grid, o, v) > 2e11 else rng.randint(1, 4)
    if call == "batch":
        # members get sizes around these (see member()); the largest grid is left to single handles
        c.update(members=rng.randint(4, 16), updates=1, v=min(v, 20), n1=1, n2=1, n3=1)
    if call == "solve":
        while flops(grid, o, c["v"]) > 3.5e11:      # a solve takes some 40 updates
            c["v"] -= 1
        v = c["v"]
        c["polish"] = "ozaki" if flops(grid, o, v) > 1e10 else rng.choice(("ozaki", "fp64"))
    return c


# ------------------------------------------------------------------------- sizes
def grid_of(c):
    return (c["n1"], c["n2"], c["n3"])


def nk(grid):
    return grid[0] * grid[1] * grid[2]


def member(c, i):
    """Grid and orbital counts of member i of a batch: uneven sizes, fixed by the case."""
    grid = ((1, 1, 1), (2, 1, 1), (2, 2, 1), (3, 1, 1))[(i * 7 + c["o"]) % 4]
    return grid, 2 + (c["o"] + 3 * i) % 7, max(4, c["v"] - 6 + (5 * i) % 13)


def flops(grid, o, v):
    """Real operations of one residual: the ladder and hole-hole sums packed by
    antisymmetry, the two ring sums, the terms in t1 (8 per complex multiply-add)."""
    n = nk(grid)
    return 8.0 * (n ** 4 * (2.0 * (o * v) ** 3 + o ** 2 * v ** 4 / 4.0 + 2.0 * o ** 4 * v ** 2 / 4.0)
                  + n ** 3 * (o * v ** 3 * (2.0 * o + v) + 4.0 * o ** 3 * v ** 2 + o ** 2 * v ** 3))


def sizes(grid, o, v):
    n = {"o": o, "v": v}
    k = nk(grid)
    return {b: k ** 3 * math.prod(n[x] for x in b) for b in BLOCKS}


def one_problem(c, grid, o, v):
    """(bytes of the inputs, bytes of the amplitudes, operations of a residual)."""
    el = 16 if c["ints"] == "c128" else 8
    k = nk(grid)
    return (float(el * sum(sizes(grid, o, v).values()) + 16 * k * (o + v) ** 2),
            16.0 * (k * o * v + k ** 3 * (o * v) ** 2), flops(grid, o, v))


def work(c):
    if c["call"] == "batch":
        got = [one_problem(c, *member(c, i)) for i in range(c["members"])]
    else:
        got = [one_problem(c, grid_of(c), c["o"], c["v"])]
    ints, amps, ops = (sum(x[k] for x in got) for k in range(3))
    if c["call"] == "energy":
        el = 16 if c["ints"] == "c128" else 8
        n2 = sizes(grid_of(c), c["o"], c["v"])["oovv"]
        return {"bytes": n2 * (16.0 + el), "flops": 8.0 * n2}
    times = {"residual": 1, "iterate": c.get("updates", 1), "batch": c.get("updates", 1),
             "solve": SOLVE_ITERATIONS}[c["call"]]
    return {"bytes": times * ints + 2 * amps, "flops": times * ops}


# ------------------------------------------------------------------------- inputs
def k_tables(grid):
    """ks[kp, kq, kr] = kp + kq - kr and neg[k] = -k on the grid, flat indices."""
    ax = [torch.arange(n) for n in grid]
    co = torch.stack(torch.meshgrid(*ax, indexing="ij"), -1).reshape(-1, 3)
    n = torch.tensor(grid)
    flat = lambda x: ((x[..., 0] % n[0]) * n[1] + x[..., 1] % n[1]) * n[2] + x[..., 2] % n[2]  # noqa: E731
    ks = flat(co[:, None, None] + co[None, :, None] - co[None, None, :])
    return ks.cuda(), flat(-co).cuda()


def raw(shape, gen, neg, time_reversal):
    n = shape[0]
    x = torch.randn(shape, dtype=torch.complex128, device="cuda", generator=gen)
    if time_reversal:
        if bool((neg.cpu() == torch.arange(n)).all()):
            x.imag.zero_()
            x *= math.sqrt(2.0)
        else:
            x = (x + x[neg][:, neg][:, :, neg].conj()) / math.sqrt(2.0)
    return x


def swap_bra(x):
    return x.transpose(0, 1).transpose(3, 4)


def swap_ket(x, ks):
    n = x.shape[0]
    k = torch.arange(n, device="cuda")
    return x[k[:, None, None], k[None, :, None], ks].transpose(5, 6)


def adjoint(x, ks):
    """conj <rs||pq> as a block [kp, kq, kr][p, q, r, s]."""
    n = x.shape[0]
    k = torch.arange(n, device="cuda")
    y = x[k[None, None, :], ks, k[:, None, None]]                 # [kp, kq, kr] = x[kr, ks, kp][r, s, p, q]
    return y.permute(0, 1, 2, 5, 6, 3, 4).conj()


def antisymmetric(shape, gen, ks, neg, time_reversal, bra, ket):
    """A random block of unit standard deviation, antisymmetric in its first / last pair."""
    x = raw(shape, gen, neg, time_reversal)
    if bra:
        x = x - swap_bra(x)
        x *= math.sqrt(0.5)
    if ket:
        x = x - swap_ket(x, ks)
        x *= math.sqrt(0.5)
    return x


def inputs(c, grid, o, v, seed):
    """The arrays a program hands to the library: Fock blocks and six integral blocks."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    ks, neg = k_tables(grid)
    n, dim, tr = nk(grid), {"o": o, "v": v}, c["time_reversal"]
    k = torch.arange(n, device="cuda")
    dt = torch.complex128 if c["ints"] == "c128" else torch.complex64
    out = {}
    for b in BLOCKS:
        shape = (n, n, n) + tuple(dim[x] for x in b)
        x = antisymmetric(shape, gen, ks, neg, tr, b[0] == b[1], b[2] == b[3])
        if b in ("oooo", "vvvv"):
            x = x + adjoint(x, ks)
            x *= math.sqrt(0.5)
        if b == "ovvo":
            # conj <ov||vo>: the adjoint with both pairs swapped, [kp,kq,kr] = x[ks,kr,kq][s,r,q,p]
            y = x[ks, k[None, None, :], k[None, :, None]]
            x = (x + y.permute(0, 1, 2, 6, 5, 4, 3).conj()) * math.sqrt(0.5)
        x *= 0.05 / n
        out[b] = x.to(dt).contiguous()
        del x

    def levels(m, lo, hi):
        e = lo + (hi - lo) * torch.rand((n, m), dtype=torch.float64, device="cuda", generator=gen)
        return 0.5 * (e + e[neg]) if tr else e

    def matrix(a, b):
        x = torch.randn((n, a, b), dtype=torch.complex128, device="cuda", generator=gen) * c["fock"]
        return (x + x[neg].conj()) * 0.5 if tr else x

    for name, m, lo, hi in (("f_oo", o, -1.5, -0.5), ("f_vv", v, 0.5, 2.5)):
        x = matrix(m, m)
        x = 0.5 * (x + x.transpose(1, 2).conj())
        x.diagonal(dim1=1, dim2=2).copy_(levels(m, lo, hi))
        out[name] = x.contiguous()
    out["f_ov"] = matrix(o, v).contiguous()
    return out


def amplitudes(c, grid, o, v, seed):
    """t1 and an antisymmetric t2 of the size they have in a solve."""
    gen = torch.Generator(device="cuda").manual_seed(seed + 7919)
    ks, neg = k_tables(grid)
    n = nk(grid)
    t2 = antisymmetric((n, n, n, o, o, v, v), gen, ks, neg, c["time_reversal"], True, True) * (0.015 / n)
    t1 = torch.randn((n, o, v), dtype=torch.complex128, device="cuda", generator=gen) * 0.01
    if c["time_reversal"]:
        t1 = (t1 + t1[neg].conj()) * math.sqrt(0.5)
    return t1.contiguous(), t2.contiguous()


# ------------------------------------------------------------------------- the calls
def prepare(c, seed):
    if c["call"] == "batch":
        problems, t = [], []
        for i in range(c["members"]):
            grid, o, v = member(c, i)
            problems.append((grid, o, v, inputs(c, grid, o, v, seed * 64 + i)))
            t.append(amplitudes(c, grid, o, v, seed * 64 + i))
        solver = binding.BatchSolver(problems, precision=PRECISION[c["form"]], diis_depth=DIIS, conv_tol=0.0)
        solver.iterate(2)           # the first iteration chooses the shapes of the launches
        handles = []
        for i in range(c["members"]):
            h = ctypes.c_void_p()
            binding.check(solver.lib.ccsd_batch_member(solver.h, i, ctypes.byref(h)), "ccsd_batch_member")
            handles.append(h)
        return {"case": c, "solver": solver, "handles": handles, "t": t,
                "out": [[torch.empty_like(t1), torch.empty_like(t2)] for t1, t2 in t]}
    grid, o, v = grid_of(c), c["o"], c["v"]
    more = {}
    if c["call"] == "solve":
        more = dict(polish_precision=PRECISION[c["polish"]], polish_iters=40, mixed_tol=1e-7, conv_tol=SOLVE_TOL,
                    max_iter=80)
    solver = binding.Solver(grid, o, v, inputs(c, grid, o, v, seed * 64), precision=PRECISION[c["form"]],
                            diis_depth=DIIS if c["call"] != "residual" else 0, **more)
    t1, t2 = amplitudes(c, grid, o, v, seed * 64)
    s = {"case": c, "solver": solver, "t1": t1, "t2": t2}
    if c["call"] == "solve":
        t1.zero_()
        t2.zero_()
    if c["call"] == "energy":
        solver.set_amplitudes(t1, t2)
    if c["call"] != "energy":
        s["o1"], s["o2"] = torch.empty_like(t1), torch.empty_like(t2)
    return s


def run(s):
    c, solver = s["case"], s["solver"]
    call = c["call"]
    if call == "residual":
        solver.residual(s["t1"], s["t2"], s["o1"], s["o2"])
        return [s["o1"], s["o2"]]
    if call == "energy":
        return [np.array([solver.energy()])]
    if call == "batch":
        for h, (t1, t2) in zip(s["handles"], s["t"]):
            binding.check(solver.lib.ccsd_set_amplitudes(h, t1.data_ptr(), t2.data_ptr()), "ccsd_set_amplitudes")
        solver.iterate(c["updates"])
        for i, (t1, t2) in enumerate(s["out"]):
            solver.member_amplitudes(i, t1, t2)
        return s["out"]
    # a program that starts from its own amplitudes (a checkpoint, a neighbouring geometry, zero)
    solver.set_amplitudes(s["t1"], s["t2"])
    if call == "iterate":
        solver.iterate(c["updates"])
    else:
        solver.solve()
    solver.get_amplitudes(s["o1"], s["o2"])
    return [s["o1"], s["o2"], np.array([solver.energy()])]


# ------------------------------------------------------------------------- 64 bits
EXACT_VVVV = 9e9                # bytes of a dense <ab||ef> that exact() still forms,
EXACT_FLOPS = 1.5e13            # and operations (about 15 s)


def exact(c, seed):
    grid, o, v = grid_of(c), c["o"], c["v"]
    n = nk(grid)
    if c["call"] == "batch":
        return [exact_one(c, *member(c, i), seed * 64 + i)[:2] for i in range(c["members"])]
    if c["call"] == "energy":
        t1, t2 = amplitudes(c, grid, o, v, seed * 64)
        a = inputs(c, grid, o, v, seed * 64)
        same = torch.arange(n, device="cuda")
        e = (a["f_ov"] * t1).sum() + 0.25 * (a["oovv"].to(torch.complex128) * t2).sum()
        for i in range(n):
            # <i ki j kj||a ki b kj> t_i^a t_j^b
            g = a["oovv"][i, same, i].to(torch.complex128)        # [kj][i, j, a, b]
            e = e + 0.5 * torch.einsum("kijab,ia,kjb->", g, t1[i], t1)
        return [(e / n).reshape(1).cpu().numpy()]
    d = 8.0 * (n * o) ** 2 * (n * v) ** 3 * (n * v + 5.0 * n * o)
    passes = {"residual": 1, "iterate": c.get("updates", 1), "solve": SOLVE_ITERATIONS}[c["call"]]
    if 16.0 * (n * v) ** 4 > EXACT_VVVV or d * passes > EXACT_FLOPS:
        return None
    return exact_one(c, grid, o, v, seed * 64)


def exact_one(c, grid, o, v, seed):
    p = Dense(c, grid, o, v, seed)
    t1, t2 = amplitudes(c, grid, o, v, seed)
    t1, t2 = p.dense1(t1), p.dense2(t2)
    if c["call"] == "residual":
        r1, r2 = p.residual(t1, t2)
        return [p.blocks1(r1), p.blocks2(r2)]
    if c["call"] == "solve":
        t1, t2 = p.solve(torch.zeros_like(t1), torch.zeros_like(t2), 200, 1e-13)
    else:
        t1, t2 = p.solve(t1, t2, c["updates"], 0.0)
    return [p.blocks1(t1), p.blocks2(t2), (p.energy(t1, t2) / p.n).reshape(1).cpu().numpy()]


class Dense:
    """The same problem over all spin orbitals (k, p) at once: the textbook spin-orbital
    CCSD equations (Stanton, Gauss, Watts and Bartlett, J. Chem. Phys. 94, 4334 (1991))
    in complex128, the Fock diagonal kept inside F."""

    def __init__(self, c, grid, o, v, seed):
        self.grid, self.o, self.v = grid, o, v
        self.n = nk(self.grid)
        self.ks = k_tables(self.grid)[0].cpu().tolist()
        a = inputs(c, grid, o, v, seed)
        self.g = {}
        for b in BLOCKS:
            self.g[b] = self.scatter(a.pop(b), b)
        self.foo, self.fvv, self.fov = (torch.zeros((self.n * x, self.n * y), dtype=torch.complex128, device="cuda")
                                        for x, y in ((self.o, self.o), (self.v, self.v), (self.o, self.v)))
        for k in range(self.n):
            for f, name, x, y in ((self.foo, "f_oo", self.o, self.o), (self.fvv, "f_vv", self.v, self.v),
                                  (self.fov, "f_ov", self.o, self.v)):
                f[k * x:(k + 1) * x, k * y:(k + 1) * y] = a[name][k]
        eo, ev = self.foo.diagonal().real, self.fvv.diagonal().real
        self.d1 = eo[:, None] - ev[None, :]
        self.d2 = eo[:, None, None, None] + eo[None, :, None, None] - ev[None, None, :, None] - ev

    def places(self, cls):
        m = [self.o if x == "o" else self.v for x in cls]
        for p in range(self.n):
            for q in range(self.n):
                for r in range(self.n):
                    at = (p, q, r, self.ks[p][q][r])
                    yield p, q, r, tuple(slice(k * s, (k + 1) * s) for k, s in zip(at, m))

    def scatter(self, x, cls):
        m = [self.n * (self.o if y == "o" else self.v) for y in cls]
        out = torch.zeros(m, dtype=torch.complex128, device="cuda")
        for p, q, r, at in self.places(cls):
            out[at] = x[p, q, r].to(torch.complex128)
        return out

    def dense2(self, t2):
        return self.scatter(t2, "oovv")

    def dense1(self, t1):
        out = torch.zeros_like(self.fov)
        for k in range(self.n):
            out[k * self.o:(k + 1) * self.o, k * self.v:(k + 1) * self.v] = t1[k]
        return out

    def blocks1(self, t1):
        return torch.stack([t1[k * self.o:(k + 1) * self.o, k * self.v:(k + 1) * self.v] for k in range(self.n)])

    def blocks2(self, t2):
        out = torch.empty((self.n,) * 3 + (self.o, self.o, self.v, self.v), dtype=torch.complex128, device="cuda")
        for p, q, r, at in self.places("oovv"):
            out[p, q, r] = t2[at]
        return out

    def residual(self, t1, t2):
        e, g, fov = torch.einsum, self.g, self.fov
        oooo, ooov, oovv, ovvo, ovvv, vvvv = (g[b] for b in BLOCKS)
        pair = e("ia,jb->ijab", t1, t1)
        pair = pair - pair.transpose(2, 3)
        tau, taut = t2 + pair, t2 + 0.5 * pair
        fae = self.fvv - 0.5 * e("me,ma->ae", fov, t1) + e("mf,mafe->ae", t1, ovvv) \
            - 0.5 * e("mnaf,mnef->ae", taut, oovv)
        fmi = self.foo + 0.5 * e("me,ie->mi", fov, t1) + e("ne,mnie->mi", t1, ooov) \
            + 0.5 * e("inef,mnef->mi", taut, oovv)
        fme = fov + e("nf,mnef->me", t1, oovv)
        x = e("je,mnie->mnij", t1, ooov)
        wmnij = oooo + x - x.transpose(2, 3) + 0.5 * e("ijef,mnef->mnij", tau, oovv)
        # <mb||ej> + t_j^f <mb||ef> - t_n^b <mn||ej> - (t_jn^fb / 2 + t_j^f t_n^b) <mn||ef>
        w = ovvo + e("jf,mbef->mbej", t1, ovvv) + e("nb,mnje->mbej", t1, ooov) \
            - e("jnfb,mnef->mbej", 0.5 * t2 + e("jf,nb->jnfb", t1, t1), oovv)
        r1 = fov.conj() + e("ie,ae->ia", t1, fae) - e("ma,mi->ia", t1, fmi) + e("imae,me->ia", t2, fme) \
            + e("nf,nafi->ia", t1, ovvo) + 0.5 * e("imef,maef->ia", t2, -ovvv) - 0.5 * e("mnae,mnie->ia", t2, ooov)
        z = e("imae,mbej->ijab", t2, w) - e("ie,ma,mbej->ijab", t1, t1, ovvo)
        za = e("ijae,be->ijab", t2, fae - 0.5 * e("mb,me->be", t1, fme)) - e("ma,ijmb->ijab", t1, ooov.conj())
        zi = e("imab,mj->ijab", t2, fmi + 0.5 * e("je,me->mj", t1, fme)) + e("ie,jeab->ijab", t1, ovvv.conj())
        lad = e("ijef,abef->ijab", tau, vvvv)
        # - P(ab) t_m^b <am||ef> = P(ab) t_m^b <ma||ef>, contracted with tau first
        y = e("ijef,maef->ijma", tau, ovvv)
        y = e("ijma,mb->ijab", y, t1)
        z = z - z.transpose(2, 3)
        z = z - z.transpose(0, 1)
        r2 = oovv.conj() + 0.5 * e("mnab,mnij->ijab", tau, wmnij) + 0.5 * (lad + y - y.transpose(2, 3)) + z \
            + za - za.transpose(2, 3) - zi + zi.transpose(0, 1)
        return r1, r2

    def energy(self, t1, t2):
        pair = torch.einsum("ia,jb->ijab", t1, t1)
        return (self.fov * t1).sum() + 0.25 * (self.g["oovv"] * t2).sum() + 0.5 * (self.g["oovv"] * pair).sum()

    def solve(self, t1, t2, updates, tol):
        """Updates t <- t + R / D with Pulay's DIIS (J. Comput. Chem. 3, 556 (1982)) over the last DIIS."""
        xs, es = [], []
        for _ in range(updates):
            r1, r2 = self.residual(t1, t2)
            if max(float(r1.abs().max()), float(r2.abs().max())) < tol:
                break
            u = torch.cat([(r1 / self.d1).reshape(-1), (r2 / self.d2).reshape(-1)])
            xs = (xs + [torch.cat([t1.reshape(-1), t2.reshape(-1)]) + u])[-DIIS:]
            es = (es + [u])[-DIIS:]
            m = len(xs)
            x = xs[-1]
            if m > 1:
                b = -np.ones((m + 1, m + 1))
                b[m, m] = 0.0
                for i in range(m):
                    for j in range(m):
                        b[i, j] = float(torch.vdot(es[i], es[j]).real)
                s = 1.0 / np.abs(b[:m, :m]).max()
                b[:m, :m] *= s
                co = np.linalg.solve(b, np.concatenate([np.zeros(m), [-1.0]]))[:m]
                x = sum(float(f) * y for f, y in zip(co, xs))
            t1, t2 = x[:t1.numel()].reshape(t1.shape), x[t1.numel():].reshape(t2.shape)
        return t1, t2
