"""The launch paths of small levels against the FP64 oracle, at the sizes where
each path begins, ends or degenerates: the FP64 cluster cycle of scalar
equations (mg_fas.cu), the tabulated FP64 coarsest vector solve
(mg_coarse.cuh), the FP32 correction cycle on a cluster (mg_clus.cu), the
integer stencils of Cartesian levels (mg_cart.cu), the batch's launch shapes
and the one-launch divergence norms.

FP64 solves follow the oracle's cycles: the count within one, every field
within 1e-9 at a converged relative residual of 1e-10, as in the solver-level
parity tests.  Mixed solves reach the same discrete solution by other
iterates: both sides converge to 1e-11, which leaves a factor 50 for the
response of the smoothest modes (2 x 50 x 1e-11 = 1e-9)."""
import threading

import numpy as np
import pytest

import oracle.oracle as o

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PI = np.pi
BOX = {"sph": ([0.0, 0.0, 0.0], [30.0, PI, 2 * PI]), "cyl": ([0.0, -30.0, 0.0], [30.0, 34.0, 2 * PI]),
       "cart": ([-30.0, -25.0, -20.0], [34.0, 27.0, 31.0]),
       "cube": ([-1.0] * 3, [1.0] * 3)}  # equal spacings on equal sizes


@pytest.fixture(scope="module")
def mg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2012_07322_gb300 import mg as m
    m.lib()
    return m


def dev(a):
    return torch.from_numpy(np.array(a, dtype=np.float64, copy=True)).cuda()


def host(t):
    return t.detach().cpu().numpy()


def solve_pair(mg, geom, n, kind, bc, precision, nu, tol, accel=0, scale=1.0):
    """The same random problem through the oracle and through the GPU."""
    lo, hi = BOX[geom][0][:len(n)], BOX[geom][1][:len(n)]
    geom = "cart" if geom == "cube" else geom
    kw = dict(tol=tol, max_cycles=1000, nu1=nu[0], nu2=nu[1], stall_window=0)
    d = o.desc(geom, n, lo, hi, accel_depth=8 if accel else 0, **kw)
    gd = mg.grid_desc(geom, n, lo, hi, precision=precision, accel_depth=accel, **kw)
    rng = np.random.default_rng(sum(n) + len(kind))
    h = mg.Hierarchy(gd)
    zero = lambda: torch.zeros(o.shape(d), dtype=torch.float64, device="cuda")
    try:
        if kind == "vec":
            f = [scale * rng.standard_normal(o.shape(d)) for _ in range(3)]
            V = [np.zeros(o.shape(d)) for _ in range(3)]
            ro = o.solve_vector(d, bc, f, V)
            Vt = [zero() for _ in range(3)]
            rg = mg.mg_solve_vector(h, bc, [dev(x) for x in f], Vt)
            return ro, rg, np.stack(V), np.stack([host(x) for x in Vt])
        if kind == "psi":
            args = dict(U=rng.uniform(0, 1e-3, o.shape(d)), A2=rng.uniform(0, 1e-4, o.shape(d)))
        else:
            args = dict(f=scale * rng.standard_normal(o.shape(d)))
            if kind == "lin_c":
                args["c"] = rng.uniform(0, 0.01, o.shape(d))
            if bc == "neumann":
                args["f"] -= args["f"].mean()
        k = "psi" if kind == "psi" else "lin"
        u = np.zeros(o.shape(d))
        ro = o.solve_scalar(d, k, bc, u, zero_mean=bc == "neumann", **args)
        ut = zero()
        rg = mg.mg_solve_scalar(h, k, bc, ut, zero_mean=bc == "neumann", **{q: dev(v) for q, v in args.items()})
        return ro, rg, u, host(ut)
    finally:
        h.close()


def check(ro, rg, want, got, cycles):
    assert ro["status"] == "ok" and rg["status"] == "ok"
    if cycles:
        assert abs(rg["cycles"] - ro["cycles"]) <= 1, (rg["cycles"], ro["cycles"])
    assert np.abs(got - want).max() <= 1e-9 * np.abs(want).max()


# 4096 and 2048 cells (the cluster's largest level and one below), 256 cells
# (its smallest), 128 and fewer (one block), wide and flat coarsest levels
@pytest.mark.parametrize("geom,n,kind,bc,nu", [
    ("sph", [64, 32], "psi", "robin", (2, 2)),
    ("sph", [32, 16, 8], "psi", "robin", (1, 2)),
    ("sph", [16, 8], "lin_c", "dirichlet", (2, 1)),
    ("sph", [16, 16], "psi", "robin", (3, 1)),
    ("cyl", [32, 64], "lin_c", "robin", (2, 2)),
    ("cyl", [16, 16, 16], "lin", "dirichlet", (1, 1)),
    ("cyl", [8, 16], "psi", "robin", (2, 0)),
    ("cart", [16, 16, 16], "lin", "robin", (2, 2)),
    ("cart", [32, 8], "lin", "neumann", (2, 2)),
    ("cart", [64, 64], "psi", "dirichlet", (0, 2)),
])
def test_fp64_scalar_small_levels(mg, geom, n, kind, bc, nu):
    check(*solve_pair(mg, geom, n, kind, bc, "fp64", nu, 1e-10), cycles=True)


# coarsest systems of 24 to 192 unknowns, two and three dimensions, and a
# level below the warp size
@pytest.mark.parametrize("geom,n,bc", [
    ("sph", [8, 4], "dirichlet"), ("sph", [32, 16, 8], "dirichlet"), ("cyl", [16, 64], "dirichlet"),
    ("cyl", [8, 8, 8], "dirichlet"), ("cart", [16, 8], "dirichlet"), ("cart", [16, 16, 8], "robin"),
])
def test_fp64_vector_small_levels(mg, geom, n, bc):
    check(*solve_pair(mg, geom, n, "vec", bc, "fp64", (2, 2), 1e-10), cycles=True)


# first levels of 2048 and 8192 cells, levels either side of the one-block
# ones (512 cells), a coarser level of the cluster below a launched one
@pytest.mark.parametrize("geom,n,kind,bc,nu", [
    ("sph", [64, 32], "psi", "robin", (2, 2)),
    ("sph", [64, 32], "vec", "dirichlet", (1, 2)),
    ("sph", [32, 16, 16], "psi", "robin", (2, 1)),
    ("sph", [32, 16, 16], "vec", "dirichlet", (2, 2)),
    ("sph", [32, 32, 16], "lin_c", "robin", (2, 2)),
    ("cyl", [64, 128], "lin_c", "robin", (2, 2)),
    ("cyl", [64, 128], "vec", "dirichlet", (2, 2)),
    ("cyl", [16, 16, 16], "vec", "dirichlet", (2, 2)),
    ("cart", [16, 16, 16], "lin", "robin", (2, 2)),
    ("cart", [128, 32], "lin", "dirichlet", (2, 2)),
    ("cart", [16, 16, 16], "vec", "dirichlet", (2, 2)),
    ("cart", [64, 64], "vec", "dirichlet", (2, 2)),
    ("cart", [32, 64], "lin", "neumann", (2, 2)),
])
def test_fp32_cycle_on_a_cluster(mg, geom, n, kind, bc, nu):
    check(*solve_pair(mg, geom, n, kind, bc, "mixed", nu, 1e-11, accel=8), cycles=False)


# fields near the ends of the exponent range go the stencils' other way; a
# linear equation scales exactly with its right-hand side
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("geom,exponent", [("cube", -80), ("cube", 60), ("cart", 60)])
def test_cartesian_stencils_scale_with_the_field(mg, precision, geom, exponent):
    n = [32, 32, 32]
    one = solve_pair(mg, geom, n, "lin", "robin", precision, (2, 2), 1e-10)
    far = solve_pair(mg, geom, n, "lin", "robin", precision, (2, 2), 1e-10, scale=2.0 ** exponent)
    check(*one, cycles=precision == "fp64")
    assert far[1]["status"] == "ok"
    assert np.abs(far[3] * 2.0 ** -exponent - one[3]).max() <= 1e-9 * np.abs(one[3]).max()


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_cartesian_stencils_carry_bad_values(mg, bad):
    gd = mg.grid_desc("cart", [32, 32, 32], [-1.0] * 3, [1.0] * 3, max_cycles=5)
    h = mg.Hierarchy(gd)
    f = np.zeros((32, 32, 32))
    f[3, 4, 5] = bad
    u = torch.zeros((32, 32, 32), dtype=torch.float64, device="cuda")
    rg = mg.mg_solve_scalar(h, "lin", "dirichlet", u, f=dev(f), allow=tuple(range(8)))
    h.close()
    assert rg["status"] != "ok"


# one cell, one row, sizes around a block and no powers of two
@pytest.mark.parametrize("n", [[1, 1], [3, 5, 7], [257, 3], [31, 33, 2], [1, 64, 5]])
def test_divergence_norms_of_odd_grids(mg, n):
    rng = np.random.default_rng(sum(n))
    B = [rng.standard_normal(tuple(reversed(n))) for _ in n]
    lo, hi = [0.0] * len(n), [0.5 + 0.25 * k for k in range(len(n))]
    div = 0.0
    for d, b in enumerate(B):
        ax = len(n) - 1 - d
        p = np.pad(b, [(1, 1) if a == ax else (0, 0) for a in range(len(n))], mode="edge")
        up, dn = np.take(p, range(2, n[d] + 2), ax), np.take(p, range(n[d]), ax)
        div = div + (up - dn) / (2 * (hi[d] - lo[d]) / n[d])
    st, mx, l2 = mg.mg_divb_norms_noalloc([dev(b) for b in B], lo, hi)
    # a sum of three differences of O(1) values over the spacing, ~10 roundings of its largest term
    tiny = 1e-14 * max(n[d] / (hi[d] - lo[d]) for d in range(len(n)))
    assert st == mg.MG_OK
    assert abs(mx - np.abs(div).max()) <= tiny and abs(l2 - np.sqrt(np.mean(div ** 2))) <= tiny


# the mixing sums are taken in the same parts whatever the team, so a problem's
# fields and cycles do not depend on the launch shape (chosen or given): bit for bit
@pytest.mark.parametrize("team,team_cells", [(1, 0), (2, 2048), (8, 8192)])
def test_batch_does_not_depend_on_the_team(mg, team, team_cells):
    from paper_2012_07322_gb300 import inputs
    ps = []
    for geom, n in (("sph", [64, 32]), ("cyl", [64, 128])):
        if geom == "sph":
            S = inputs.rotating_polytrope_sph2d(n[0], n[1], 100.0, 1e-3, 10.0, axis_ratio=0.8, omega=0.02)
            lo, hi = [0.0, 0.0], [100.0, PI]
        else:
            S = inputs.rotating_polytrope_cyl(n, 100.0, 1e-3, 10.0, axis_ratio=0.8, omega=0.02)
            lo, hi = [0.0, -100.0], [100.0, 100.0]
        h = mg.Hierarchy(mg.grid_desc(geom, n, lo, hi, precision="mixed", tol=1e-10, accel_depth=16, stall_window=0))
        one = lambda: torch.ones(S[0].shape, dtype=torch.float64, device="cuda")
        ps.append((h, dev(S[0]), dev(S[1]), [dev(x) for x in S[2]], one(), one(), [one() for _ in range(3)],
                   [one() for _ in range(3)]))

    def solve(**shape):
        for p in ps:
            for t in (p[4], p[5]):
                t.fill_(1.0)
            for t in p[6] + p[7]:
                t.zero_()
        reps, b = mg.mg_solve_cfc_batch(ps, **shape)
        assert b["status"] == "ok"
        return ([t.clone() for p in ps for t in [p[4], p[5]] + p[6] + p[7]],
                [r[k]["cycles"] for r in reps for k in ("X", "psi", "alphapsi", "beta")])

    want, cycles = solve()
    got, again = solve(team=team, team_cells=team_cells)
    for p in ps:
        p[0].close()
    assert again == cycles
    assert all(torch.equal(a, b) for a, b in zip(got, want))


# ---- order of the cluster cycles: a value is replaced only behind every read of it


class Busy:
    """Another hierarchy solving on its own stream: blocks of the measured cycle are held back at places that change
    from run to run."""

    def __init__(self, mg):
        self.mg, self.stop = mg, threading.Event()
        self.thread = threading.Thread(target=self.loop)

    def loop(self):
        mg, n = self.mg, [64, 64, 32]
        with torch.cuda.stream(torch.cuda.Stream()):
            h = mg.Hierarchy(mg.grid_desc("cart", n, BOX["cart"][0], BOX["cart"][1], precision="mixed", tol=1e-10))
            f = torch.ones(tuple(reversed(n)), dtype=torch.float64, device="cuda")
            u = torch.zeros_like(f)
            while not self.stop.is_set():
                u.zero_()
                mg.mg_solve_scalar(h, "lin", "dirichlet", u, f=f)
            h.close()

    def __enter__(self):
        self.thread.start()

    def __exit__(self, *exc):
        self.stop.set()
        self.thread.join()


def first_cycles(mg, geom, n, kind, bc, precision, nu, cycles, repeats):
    """The iterate behind some cycles from zero, by the oracle (once) and by the GPU (repeated beside other work)."""
    lo, hi = BOX[geom][0][:len(n)], BOX[geom][1][:len(n)]
    kw = dict(tol=1e-14, max_cycles=cycles, nu1=nu[0], nu2=nu[1], stall_window=0)
    d = o.desc(geom, n, lo, hi, **kw)
    shape = (3,) + o.shape(d) if kind == "vec" else o.shape(d)
    rng = np.random.default_rng(sum(n))
    want = np.zeros(shape)
    if kind == "vec":
        f = rng.standard_normal(shape)
        o.solve_vector(d, bc, list(f), list(want))
    else:
        args = dict(f=rng.standard_normal(shape), c=rng.uniform(0, 0.01, shape))
        if kind == "psi":
            args = dict(U=rng.uniform(0, 1e-3, shape), A2=rng.uniform(0, 1e-4, shape))
        o.solve_scalar(d, kind, bc, want, **args)
        args = {k: dev(v) for k, v in args.items()}
    h = mg.Hierarchy(mg.grid_desc(geom, n, lo, hi, precision=precision, **kw))
    got = []
    with Busy(mg):
        for _ in range(repeats):
            u = torch.zeros(shape, dtype=torch.float64, device="cuda")
            if kind == "vec":
                mg.mg_solve_vector(h, bc, list(dev(f)), list(u), allow=tuple(range(8)))
            else:
                mg.mg_solve_scalar(h, kind, bc, u, allow=tuple(range(8)), **args)
            got.append(u)
    h.close()
    return want, got


# A right-hand side formed from half-swept values is off by the size of the
# correction (1e-3 and more); a few hundred passes of a contraction carry
# rounding errors of a few 1e-16 each, and the oracle's coarsest solve may stop
# at a residual of 1e-12: 1e-10 in all.
@pytest.mark.parametrize("geom,n,kind,bc,nu", [
    ("sph", [64, 32], "psi", "robin", (2, 2)), ("sph", [32, 16, 8], "psi", "robin", (1, 2)),
    ("cyl", [32, 64], "lin", "robin", (2, 1)), ("cart", [16, 16, 16], "lin", "robin", (2, 2)),
    ("cart", [16, 8], "lin", "dirichlet", (2, 2)),
])
def test_fp64_scalar_cycles_in_order(mg, geom, n, kind, bc, nu):
    want, got = first_cycles(mg, geom, n, kind, bc, "fp64", nu, 3, 50)
    assert np.abs(host(got[0]) - want).max() <= 1e-10 * np.abs(want).max()
    assert all(torch.equal(g, got[0]) for g in got)


# levels on all blocks and on the first one; ghosts from across the origin, the
# axis and the poles, which other blocks' cells are the sources of
@pytest.mark.parametrize("geom,n,nu", [
    ("sph", [64, 32], (2, 2)), ("sph", [32, 16, 16], (1, 1)), ("cyl", [64, 128], (2, 2)), ("cyl", [16, 16, 16], (0, 2)),
    ("cart", [64, 64], (2, 0)),
])
def test_fp32_vector_cycles_in_order(mg, geom, n, nu):
    _, got = first_cycles(mg, geom, n, "vec", "dirichlet", "mixed", nu, 8, 50)
    assert bool(torch.isfinite(got[0]).all()) and float(got[0].abs().max()) > 0.0
    assert all(torch.equal(g, got[0]) for g in got)


# at least two levels on all blocks, one level above the first block's, none;
# tolerance as for the scalar cycles
@pytest.mark.parametrize("geom,n,nu", [
    ("sph", [32, 16, 8], (2, 2)), ("sph", [16, 8, 8], (1, 2)), ("cyl", [32, 64], (2, 2)), ("cyl", [16, 16, 16], (2, 1)),
    ("cart", [16, 16, 16], (2, 2)), ("cart", [16, 8], (2, 2)),
])
def test_fp64_vector_cycles_in_order(mg, geom, n, nu):
    want, got = first_cycles(mg, geom, n, "vec", "dirichlet", "fp64", nu, 3, 50)
    assert np.abs(host(got[0]) - want).max() <= 1e-10 * np.abs(want).max()
    assert all(torch.equal(g, got[0]) for g in got)


# two threads at once (which the call's description rules out) may get each
# other's norms; the calls behind them get their own
def test_divergence_norms_after_overlapping_calls(mg):
    def field(n):
        B = [dev(np.random.default_rng(n).standard_normal((n, n, n))) for _ in range(3)]
        return B, [0.0] * 3, [1.0] * 3

    fields = [field(16), field(48), field(96)]
    want = [mg.mg_divb_norms_noalloc(*f) for f in fields]
    torch.cuda.synchronize()

    def loop(f):
        s = torch.cuda.Stream()
        for _ in range(400):
            mg.mg_divb_norms_noalloc(*f, stream=s)

    threads = [threading.Thread(target=loop, args=(f,)) for f in fields]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for _ in range(3):
        assert [mg.mg_divb_norms_noalloc(*f) for f in fields] == want


# FMG starts a level from the coarser level's correction, also the level whose
# V-cycle runs on a cluster (8192 cells: the finest here).  Dropped, an FMG cycle
# is a V-cycle.  Cycles: what passes launched one by one take.
@pytest.mark.parametrize("geom,n,kind,bc,accel,cycles", [
    ("cart", [128, 64], "lin", "dirichlet", 0, 9), ("cart", [32, 16, 16], "lin", "robin", 0, 12),
    ("cart", [32, 16, 16], "vec", "dirichlet", 0, 12), ("cyl", [64, 128], "lin", "robin", 8, 6),
    ("cyl", [64, 128], "vec", "dirichlet", 8, 6),
])
def test_mixed_fmg_keeps_its_starting_guess(mg, geom, n, kind, bc, accel, cycles):
    lo, hi = BOX[geom][0][:len(n)], BOX[geom][1][:len(n)]
    shape = (3,) * (kind == "vec") + tuple(reversed(n))
    f = dev(np.random.default_rng(5).standard_normal(shape))
    took = {}
    for cycle in ("v", "fmg"):
        h = mg.Hierarchy(mg.grid_desc(geom, n, lo, hi, precision="mixed", tol=1e-10, max_cycles=100, stall_window=0,
                                      accel_depth=accel, cycle=cycle))
        u = torch.zeros(shape, dtype=torch.float64, device="cuda")
        if kind == "vec":
            took[cycle] = mg.mg_solve_vector(h, bc, list(f), list(u))["cycles"]
        else:
            took[cycle] = mg.mg_solve_scalar(h, kind, bc, u, f=f)["cycles"]
        h.close()
    assert took["fmg"] < took["v"] and took["fmg"] <= cycles


# The integer stencils hand over to the flux form where all seven values lie
# below 2^-895 or the scaled coefficient is not normal: right-hand sides that
# put the solution (2^-10 to 2^-5 of them on the unit cube) on both sides of
# the first line and below it, close to overflow, and, with cells of 2^40, on
# both sides of the second.  A linear equation scales exactly with powers of two.
@pytest.mark.parametrize("side,exponent", [(0, -888), (0, -920), (0, 1008), (44, -963)])
def test_cartesian_stencils_at_the_ends_of_the_range(mg, side, exponent):
    f = np.random.default_rng(12).standard_normal((32, 32, 32))

    def solve(side, exponent):
        h = mg.Hierarchy(mg.grid_desc("cart", [32] * 3, [-2.0 ** side] * 3, [2.0 ** side] * 3, tol=1e-10,
                                      max_cycles=100, stall_window=0))
        u = torch.zeros((32, 32, 32), dtype=torch.float64, device="cuda")
        rg = mg.mg_solve_scalar(h, "lin", "robin", u, f=dev(np.ldexp(f, exponent)))
        h.close()
        return rg, np.ldexp(host(u), -exponent - 2 * side)

    one, want = solve(0, 0)
    far, got = solve(side, exponent)
    assert abs(far["cycles"] - one["cycles"]) <= 1
    assert np.abs(got - want).max() <= 1e-9 * np.abs(want).max()


# as many planes as a launch of two-plane blocks takes, rows short enough for
# blocks of one plane: the passes run and the first cycles converge
@pytest.mark.parametrize("kind", ["lin", "vec"])
def test_fp64_passes_of_65536_planes(mg, kind):
    n = [16, 16, 65536]
    h = mg.Hierarchy(mg.grid_desc("cart", n, [0.0] * 3, [1.0, 1.0, 4096.0], tol=1e-14, max_cycles=3, stall_window=0))
    shape = (3,) * (kind == "vec") + tuple(reversed(n))
    f = torch.randn(shape, generator=torch.Generator(device="cuda").manual_seed(1), dtype=torch.float64, device="cuda")
    u = torch.zeros_like(f)
    if kind == "vec":
        rg = mg.mg_solve_vector(h, "dirichlet", list(f), list(u), allow=tuple(range(8)))
    else:
        rg = mg.mg_solve_scalar(h, "lin", "dirichlet", u, f=f, allow=tuple(range(8)))
    h.close()
    assert rg["cycles"] == 3 and rg["rel"] < 0.1
