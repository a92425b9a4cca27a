"""The work a user has this library do, case by case: single xCFC solves, divergence cleanings, composite-grid
solves, batches, a burst of server requests and the per-step divergence monitor, each through the package's public
calls, with seeded inputs and, where one is affordable, the answer in 64 bits from plain torch.

A case is a dict of plain values; "kind" selects the call:
    norms    mg_divb_norms_noalloc on a Cartesian field of any size
    psi      eq. psi alone (static star), axisymmetric 2D grids
    xcfc     the four xCFC equations of a rotating star, 2D and 3D grids
    divb     elliptic divergence cleaning, compact or exact projection
    amr      eq. psi on the two-level composite grid
    batch    independent 2D xCFC solves in one persistent launch
    serve    a burst of mixed requests through the server
"""
import math

import numpy as np
import torch

from paper_2012_07322_gb300 import mg

PI = math.pi
TOL = 1e-10
MAX_CYCLES = 1000


def listed():
    return [
        # The divergence monitor an evolution code calls every time step on a block it owns: the smallest call, any
        # block size.
        {"name": "norms_56x40x48", "kind": "norms", "n0": 56, "n1": 40, "n2": 48},
        # Initial data of one non-rotating star, the paper's plain iteration in FP64: the smallest solve, a chain of
        # small launches.
        {"name": "psi_sph_64x32_fp64", "kind": "psi", "geom": "sph", "n0": 64, "n1": 32, "precision": "fp64",
         "accel": 0},
        # A rotating star on the axisymmetric grid of a production 2D run, mixed precision: a metric update.
        {"name": "xcfc_cyl_64x128_mixed", "kind": "xcfc", "geom": "cyl", "n0": 64, "n1": 128, "n2": 0,
         "precision": "mixed"},
        # A deformed rotating star in 3D, FP64 throughout: the reference route users check the mixed one against.
        {"name": "xcfc_sph_64x32x32_fp64", "kind": "xcfc", "geom": "sph", "n0": 64, "n1": 32, "n2": 32,
         "precision": "fp64"},
        # The 3D production solve, mixed precision.
        {"name": "xcfc_sph_128x64x64_mixed", "kind": "xcfc", "geom": "sph", "n0": 128, "n1": 64, "n2": 64,
         "precision": "mixed"},
        # Cleaning one block of a magnetised run: an ordinary size.
        {"name": "divb_64_mixed", "kind": "divb", "n0": 64, "n1": 64, "n2": 64, "precision": "mixed",
         "variant": "compact"},
        # Cleaning the whole cube: every finest array is larger than the L2 cache.
        {"name": "divb_256_mixed", "kind": "divb", "n0": 256, "n1": 256, "n2": 256, "precision": "mixed",
         "variant": "compact"},
        # The same cleaning with every kernel in FP64.
        {"name": "divb_128_fp64", "kind": "divb", "n0": 128, "n1": 128, "n2": 128, "precision": "fp64",
         "variant": "compact"},
        # The exact projection (the divergence the update sees is removed entirely).
        {"name": "divb_exact_128_mixed", "kind": "divb", "n0": 128, "n1": 128, "n2": 128, "precision": "mixed",
         "variant": "exact"},
        # A star refined for r < r_max / 4 on the two-level grid, FP64.
        {"name": "amr_sph_64x32x32", "kind": "amr", "n0": 64, "n1": 32, "n2": 32},
        # A parameter scan: uneven 2D grids of rotating stars, all in one persistent launch.
        {"name": "batch_192_mixed", "kind": "batch", "count": 192, "omega": 0.02, "shapes": 3},
        # A burst of requests of different geometries and sizes on four worker slots.
        {"name": "serve_12", "kind": "serve", "count": 12, "slots": 4, "mix": 0},
    ]


def draw(rng):
    kind = rng.choice(["norms", "norms", "psi", "xcfc", "xcfc", "divb", "divb", "divb", "amr", "batch", "serve"])
    if kind == "norms":
        # any block size from 8 cells a side to the call's limit, planar and 3D
        if rng.random() < 0.25:
            return {"kind": kind, "n0": int(2 ** rng.uniform(4, 10)), "n1": int(2 ** rng.uniform(4, 10)), "n2": 0}
        return {"kind": kind, "n0": int(2 ** rng.uniform(3, 7)), "n1": int(2 ** rng.uniform(3, 7)),
                "n2": int(2 ** rng.uniform(3, 7))}
    if kind == "psi":
        geom = rng.choice(["sph", "cyl"])
        n0 = rng.choice([32, 64, 128])
        n1 = rng.choice([16, 32, 64]) if geom == "sph" else 2 * n0
        # point smoothing needs the mixing on grids that are finer in theta
        return {"kind": kind, "geom": geom, "n0": n0, "n1": n1, "precision": rng.choice(["fp64", "mixed"]),
                "accel": rng.choice([8, 12, 16])}
    if kind == "xcfc":
        shape = rng.choice([("sph", 64, 32, 0), ("sph", 128, 64, 0), ("cyl", 32, 64, 0), ("cyl", 128, 256, 0),
                            ("sph", 32, 16, 16), ("sph", 64, 32, 32), ("sph", 64, 16, 32), ("cyl", 16, 32, 8),
                            ("cyl", 32, 64, 16)])
        return {"kind": kind, "geom": shape[0], "n0": shape[1], "n1": shape[2], "n2": shape[3],
                "precision": rng.choice(["mixed", "mixed", "fp64"])}
    if kind == "divb":
        variant = rng.choice(["compact", "compact", "exact"])
        precision = rng.choice(["mixed", "mixed", "fp64"])
        top = 128 if precision == "fp64" or variant == "exact" else 256
        base = rng.choice([s for s in (32, 64, 128, 256) if s <= top])
        n = [base, base, base]
        if rng.random() < 0.5:
            n[rng.randrange(3)] = max(16, base // 2)
        return {"kind": kind, "n0": n[0], "n1": n[1], "n2": n[2], "precision": precision, "variant": variant}
    if kind == "amr":
        n0, n1, n2 = rng.choice([(32, 16, 16), (64, 32, 32), (32, 16, 0), (64, 32, 0), (64, 16, 16)])
        return {"kind": kind, "n0": n0, "n1": n1, "n2": n2}
    if kind == "batch":
        return {"kind": kind, "count": rng.randint(3, 127), "omega": rng.choice([0.0, 0.02]),
                "shapes": rng.randrange(1000)}
    return {"kind": kind, "count": rng.randint(2, 12), "slots": rng.choice([1, 2, 4, 8]), "mix": rng.randrange(1000)}


# ------------------------------------------------------------------ inputs


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _centres(n, lo, hi):
    return [lo[d] + (np.arange(n[d]) + 0.5) * (hi[d] - lo[d]) / n[d] for d in range(len(n))]


def _star(geom, n, lo, hi, rho_c, R, axis_ratio, omega, bar):
    """U~, S~ and S~_i (orthonormal components) of an n = 1 polytrope (K = 100, G = c = M_sun = 1) that rotates
    uniformly, oblate by axis_ratio, its surface deformed by a bar (m = 2) of relative amplitude `bar` in 3D."""
    c = _centres(n, lo, hi)
    three = len(n) == 3
    x = c[0].reshape((1,) * (len(n) - 1) + (-1,))
    y = c[1].reshape((1, -1, 1) if three else (-1, 1))
    ph = c[2].reshape(-1, 1, 1) if three else 0.0
    if geom == "sph":
        varpi, z = x * np.sin(y), x * np.cos(y)
    else:
        varpi, z = x + 0.0 * y, y + 0.0 * x
    shp = tuple(reversed(n))
    xi = np.sqrt((varpi / R) ** 2 * (1.0 + bar * np.cos(2.0 * ph)) + (z / (axis_ratio * R)) ** 2)
    xi = np.broadcast_to(xi, shp)
    rho = np.where(xi < 1.0, rho_c * np.sinc(np.minimum(xi, 1.0)), 0.0)
    v = omega * varpi
    w2 = 1.0 / (1.0 - v * v)
    p = 100.0 * rho * rho
    a = rho * (1.0 + 200.0 * rho) * w2
    Si = np.zeros((3,) + shp)
    Si[2] = a * v
    return a - p, a * v * v + 3.0 * p, Si


def _domain(geom, n):
    if geom == "sph":
        lo, hi = [0.0, 0.0, 0.0], [100.0, PI, 2 * PI]
    else:
        lo, hi = [0.0, -100.0, 0.0], [100.0, 100.0, 2 * PI]
    return lo[: len(n)], hi[: len(n)]


def _size(case):
    return [case[k] for k in ("n0", "n1", "n2") if case[k]]


def _draw_star(rng):
    return rng.uniform(5e-4, 2e-3), rng.uniform(8.0, 14.0)


def _psi_source(case, seed):
    n = [case["n0"], case["n1"]]
    lo, hi = _domain(case["geom"], n)
    rho_c, R = _draw_star(np.random.default_rng(seed))
    return n, lo, hi, _star(case["geom"], n, lo, hi, rho_c, R, 1.0, 0.0, 0.0)[0]


def _box(n):
    """Domain of cubic cells, the longest side [-1, 1]."""
    m = max(n)
    return [-k / m for k in n], [k / m for k in n]


def _divb_field(n, lo, hi, seed):
    """B = central curl of 16 random Fourier modes plus noise of 1e-3 of its rms (the divergence to be cleaned), as one
    (3, n2, n1, n0) tensor."""
    rng = np.random.default_rng(seed)
    k = torch.from_numpy(rng.integers(-8, 9, size=(16, 3)).astype(np.float64)).cuda()
    amp = torch.from_numpy(rng.standard_normal((3, 16))).cuda()
    ph = torch.from_numpy(rng.uniform(0, 2 * PI, 16)).cuda()
    h = [(hi[d] - lo[d]) / n[d] for d in range(3)]
    x = [lo[d] + (torch.arange(-1, n[d] + 1, dtype=torch.float64, device="cuda") + 0.5) * h[d] for d in range(3)]
    e = [PI * k[:, d, None] * x[d] for d in range(3)]
    exy = e[0][:, None, :] + e[1][:, :, None] + ph[:, None, None]
    s, c = torch.sin(exy).reshape(16, -1), torch.cos(exy).reshape(16, -1)
    sz, cz = torch.sin(e[2]), torch.cos(e[2])
    shp = tuple(m + 2 for m in reversed(n))
    A = [((amp[q, :, None] * cz).T @ s + (amp[q, :, None] * sz).T @ c).reshape(shp) for q in range(3)]
    I = slice(1, -1)
    dx = lambda F: (F[I, I, 2:] - F[I, I, :-2]) / (2 * h[0])
    dy = lambda F: (F[I, 2:, I] - F[I, :-2, I]) / (2 * h[1])
    dz = lambda F: (F[2:, I, I] - F[:-2, I, I]) / (2 * h[2])
    B = torch.stack([dy(A[2]) - dz(A[1]), dz(A[0]) - dx(A[2]), dx(A[1]) - dy(A[0])])
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    return B + torch.randn(B.shape, generator=g, dtype=torch.float64, device="cuda") * (1e-3 * B.square().mean().sqrt())


def _norms_field(case, seed):
    n = _size(case)
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    return n, torch.randn((len(n),) + tuple(reversed(n)), generator=g, dtype=torch.float64, device="cuda")


_BATCH_NR, _BATCH_NT, _BATCH_NZ = [32, 64, 128, 256], [16, 32, 64, 128], [64, 128, 256, 512]


def _batch_shapes(case):
    """Uneven grids: half spherical, half cylindrical."""
    rng = np.random.default_rng(case["shapes"])
    out = []
    for q in range(case["count"]):
        n0 = int(rng.choice(_BATCH_NR))
        out.append(("sph", [n0, int(rng.choice(_BATCH_NT))]) if q % 2 == 0 else ("cyl", [n0, int(rng.choice(_BATCH_NZ))]))
    return out


# Requests the server meets: metric solves on 2D and small 3D grids, cleanings of two block sizes.
_SERVE = [("sph", [64, 32]), ("cart", [32, 32, 32]), ("sph", [32, 16, 16]), ("cyl", [64, 128]), ("cart", [64, 64, 64]),
          ("sph", [128, 64]), ("sph", [64, 32, 32])]


def _serve_requests(case):
    rng = np.random.default_rng(case["mix"])
    order = list(range(case["count"])) if case["mix"] == 0 else [int(v) for v in rng.integers(0, len(_SERVE), case["count"])]
    return [_SERVE[q % len(_SERVE)] for q in order]


def _desc(geom, n, lo, hi, precision, accel, **kw):
    return mg.grid_desc(geom, n, lo, hi, precision=precision, tol=TOL, max_cycles=MAX_CYCLES, accel_depth=accel,
                        stall_window=0, **kw)


class _Fields:
    """Metric fields as a user's program holds them: scalars, and vectors of one (3, ...) array each."""

    def __init__(self, shp):
        new = lambda s: torch.empty(s, dtype=torch.float64, device="cuda")
        self.psi, self.alpha, self.beta, self.X = new(shp), new(shp), new((3,) + shp), new((3,) + shp)

    def flat(self):
        self.psi.fill_(1.0)
        self.alpha.fill_(1.0)
        self.beta.zero_()
        self.X.zero_()

    def args(self):
        return self.psi, self.alpha, list(self.beta), list(self.X)


def prepare(case, seed):
    kind = case["kind"]
    st = {"kind": kind}
    if kind == "norms":
        n, B = _norms_field(case, seed)
        st.update(B=list(B), lo=[0.0] * len(n), hi=[k / 64.0 for k in n])
    elif kind == "psi":
        n, lo, hi, U = _psi_source(case, seed)
        st["U"] = _dev(U)
        st["psi"] = torch.empty_like(st["U"])
        st["h"] = mg.Hierarchy(_desc(case["geom"], n, lo, hi, case["precision"], case["accel"]))
    elif kind == "xcfc":
        n = _size(case)
        lo, hi = _domain(case["geom"], n)
        rng = np.random.default_rng(seed)
        rho_c, R = _draw_star(rng)
        U, S, Si = _star(case["geom"], n, lo, hi, rho_c, R, 0.8, 0.02, rng.uniform(0.1, 0.2) if len(n) == 3 else 0.0)
        st.update(U=_dev(U), S=_dev(S), Si=list(_dev(Si)), f=_Fields(U.shape))
        st["h"] = mg.Hierarchy(_desc(case["geom"], n, lo, hi, case["precision"], 16))
    elif kind == "divb":
        n = _size(case)
        lo, hi = _box(n)
        st["B0"] = _divb_field(n, lo, hi, seed)
        st["B"] = torch.empty_like(st["B0"])
        st["h"] = mg.Hierarchy(_desc("cart", n, lo, hi, case["precision"], 0, divb=case["variant"]))
    elif kind == "amr":
        n = _size(case)
        lo, hi = _domain("sph", n)
        rho_c, R = _draw_star(np.random.default_rng(seed))
        box = [0] * len(n), [n[0] // 4] + n[1:]
        fine = [n[0] // 2] + [2 * k for k in n[1:]]
        U = _dev(_star("sph", n, lo, hi, rho_c, R, 1.0, 0.0, 0.0)[0])
        Up = _dev(_star("sph", fine, lo, [25.0] + hi[1:], rho_c, R, 1.0, 0.0, 0.0)[0])
        st.update(box=box, U=U, Up=Up, A2=torch.zeros_like(U), A2p=torch.zeros_like(Up), u=torch.empty_like(U),
                  up=torch.empty_like(Up))
        st["h"] = mg.Hierarchy(_desc("sph", n, lo, hi, "fp64", 16))
    elif kind == "batch":
        rng = np.random.default_rng(seed)
        shapes = _batch_shapes(case)
        cells = sum(n[0] * n[1] for _, n in shapes)
        new = lambda m: torch.empty(m * cells, dtype=torch.float64, device="cuda")
        # every field of the scan in one array, a problem's part contiguous in it
        st["out"] = {"psi": new(1), "alpha": new(1), "beta": new(3), "X": new(3)}
        st["problems"], at = [], 0
        for geom, n in shapes:
            lo, hi = _domain(geom, n)
            rho_c, R = _draw_star(rng)
            U, S, Si = _star(geom, n, lo, hi, rho_c, R, 0.8 if case["omega"] else 1.0, case["omega"], 0.0)
            m = n[0] * n[1]
            part = lambda t, w: t[w * at: w * (at + m)].view((w,) + U.shape)
            h = mg.Hierarchy(_desc(geom, n, lo, hi, "mixed", 16))
            st["problems"].append((h, _dev(U), _dev(S), list(_dev(Si)), part(st["out"]["psi"], 1)[0],
                                   part(st["out"]["alpha"], 1)[0], list(part(st["out"]["beta"], 3)),
                                   list(part(st["out"]["X"], 3))))
            at += m
    else:
        rng = np.random.default_rng(seed)
        st["srv"] = mg.Server(hbm_budget=16 << 30, max_slots=case["slots"], max_queue=64)
        st["reqs"] = []
        for geom, n in _serve_requests(case):
            if geom == "cart":
                lo, hi = _box(n)
                B0 = _divb_field(n, lo, hi, int(rng.integers(1 << 30)))
                st["reqs"].append((_desc(geom, n, lo, hi, "mixed", 0), None, None, None, (B0, torch.empty_like(B0))))
                continue
            lo, hi = _domain(geom, n)
            rho_c, R = _draw_star(rng)
            U, S, Si = _star(geom, n, lo, hi, rho_c, R, 0.8, 0.02, 0.15 if len(n) == 3 else 0.0)
            st["reqs"].append((_desc(geom, n, lo, hi, "mixed", 16), _dev(U), _dev(S), list(_dev(Si)), _Fields(U.shape)))
    return st


def run(st):
    kind = st["kind"]
    if kind == "norms":
        _, largest, l2 = mg.mg_divb_norms_noalloc(st["B"], st["lo"], st["hi"])
        return np.array([largest, l2])
    if kind == "psi":
        st["psi"].fill_(1.0)
        mg.mg_solve_cfc(st["h"], st["U"], None, None, st["psi"], None, None, None, psi_only=True)
        return st["psi"]
    if kind == "xcfc":
        f = st["f"]
        f.flat()
        mg.mg_solve_cfc(st["h"], st["U"], st["S"], st["Si"], *f.args())
        return {"psi": f.psi, "alpha": f.alpha, "beta": f.beta, "X": f.X}
    if kind == "divb":
        st["B"].copy_(st["B0"])
        mg.mg_clean_divB(st["h"], list(st["B"]))
        return st["B"]
    if kind == "amr":
        st["u"].zero_()
        st["up"].zero_()
        mg.mg_solve_scalar_amr(st["h"], st["box"][0], st["box"][1], "psi", "robin", st["u"], st["up"], U=st["U"],
                               A2=st["A2"], Up=st["Up"], A2p=st["A2p"])
        return {"u": st["u"], "up": st["up"]}
    if kind == "batch":
        out = st["out"]
        out["psi"].fill_(1.0)
        out["alpha"].fill_(1.0)
        out["beta"].zero_()
        out["X"].zero_()
        mg.mg_solve_cfc_batch(st["problems"], reports=False)
        return out
    srv, tickets = st["srv"], []
    for desc, U, S, Si, f in st["reqs"]:
        if U is None:
            f[1].copy_(f[0])
            tickets.append(srv.submit_divb(desc, list(f[1])))
        else:
            f.flat()
            tickets.append(srv.submit_cfc(desc, U, S, Si, *f.args()))
    for t in tickets:
        srv.wait(t)
    return [f[1] if U is None else {"psi": f.psi, "alpha": f.alpha, "beta": f.beta, "X": f.X}
            for _, U, _, _, f in st["reqs"]]


# -------------------------------------------------------------------- work

# Operations per cell of one defect-correction or FAS cycle V(2, 2): four sweeps, residual and transfers of a scalar
# equation (7-point stencil), eight sevenths of it for the coarser grids; a vector cycle has three components of
# about three times the stencil.  Cycles a multigrid of this smoother needs to 1e-10: about 12 on Cartesian grids, 40
# with mixing on curvilinear ones.
_SCALAR, _VECTOR = 5 * 16 * 8 / 7, 9 * 5 * 16 * 8 / 7


def work(case):
    kind = case["kind"]
    if kind == "norms":
        n = _size(case)
        return {"bytes": 8.0 * len(n) * math.prod(n) + 16, "flops": 12.0 * math.prod(n)}
    if kind == "psi":
        cells = case["n0"] * case["n1"]
        return {"bytes": 24.0 * cells, "flops": 40 * _SCALAR * cells}
    if kind == "xcfc":
        return _xcfc_work(math.prod(_size(case)))
    if kind == "divb":
        return _divb_work(math.prod(_size(case)))
    if kind == "amr":
        cells = math.prod(_size(case))
        cells += cells // 4 * 2 ** len(_size(case))
        return {"bytes": 32.0 * cells, "flops": 40 * _SCALAR * cells}
    parts = []
    if kind == "batch":
        parts = [_xcfc_work(n[0] * n[1]) for _, n in _batch_shapes(case)]
        if not case["omega"]:
            parts = [{"bytes": p["bytes"], "flops": 80 * _SCALAR * n[0] * n[1]}
                     for p, (_, n) in zip(parts, _batch_shapes(case))]
    else:
        parts = [(_divb_work if g == "cart" else _xcfc_work)(math.prod(n)) for g, n in _serve_requests(case)]
    return {"bytes": sum(p["bytes"] for p in parts), "flops": sum(p["flops"] for p in parts)}


def _xcfc_work(cells):
    return {"bytes": 8.0 * (5 + 8 + 8) * cells, "flops": 40 * (2 * _SCALAR + 2 * _VECTOR) * cells}


def _divb_work(cells):
    return {"bytes": 8.0 * 6 * cells, "flops": (12 * _SCALAR + 24) * cells}


# ------------------------------------------------------- answers in 64 bits


def exact(case, seed):
    """Norms, cleanings and the axisymmetric eq. psi have a direct solution that plain torch gives in seconds.  The
    deformed stars in 3D, the composite grid and whole batches have none that takes under 20 s."""
    kind = case["kind"]
    if kind == "norms":
        n, B = _norms_field(case, seed)
        div = sum(_central(B[d], len(n) - 1 - d, 1.0 / 64.0) for d in range(len(n)))
        return np.array([float(div.abs().max()), math.sqrt(float(div.square().mean()))])
    if kind == "divb":
        n = _size(case)
        lo, hi = _box(n)
        return _clean(_divb_field(n, lo, hi, seed), n, [(hi[d] - lo[d]) / n[d] for d in range(3)], case["variant"])
    if kind == "psi":
        return _psi_direct(*_psi_source(case, seed), case["geom"])
    return None


def _shift(F, ax, step, edge):
    """F moved by one cell along ax; the ghost beyond the end is the cell at distance `edge` from it."""
    n = F.shape[ax]
    idx = torch.arange(n, device=F.device) + step
    idx = torch.where(idx < 0, torch.full_like(idx, edge), torch.where(idx >= n, torch.full_like(idx, n - 1 - edge), idx))
    return F.index_select(ax, idx)


def _central(F, ax, h, edge=0):
    return (_shift(F, ax, 1, edge) - _shift(F, ax, -1, edge)) / (2 * h)


def _neumann(b, n, h):
    """Zero-mean solution of the compact Neumann Poisson problem by the cosine transform of each direction."""
    lam, q = [], []
    for d in range(3):
        i = torch.arange(n[d], dtype=torch.float64, device=b.device)
        V = torch.cos(PI * i[:, None] * (i[None, :] + 0.5) / n[d]) * math.sqrt(2.0 / n[d])
        V[0] *= math.sqrt(0.5)
        q.append(V)
        lam.append(-4.0 * torch.sin(PI * i / (2 * n[d])) ** 2 / h[d] ** 2)
    t = torch.einsum("kz,zyx->kyx", q[2], b)
    t = torch.einsum("jy,kyx->kjx", q[1], t)
    t = torch.einsum("ix,kjx->kji", q[0], t)
    L = lam[2][:, None, None] + lam[1][None, :, None] + lam[0][None, None, :]
    L[0, 0, 0] = 1.0
    t = t / L
    t[0, 0, 0] = 0.0
    t = torch.einsum("ix,kji->kjx", q[0], t)
    t = torch.einsum("jy,kjx->kyx", q[1], t)
    return torch.einsum("kz,kyx->zyx", q[2], t)


def _clean(B, n, h, variant):
    div = sum(_central(B[d], 2 - d, h[d]) for d in range(3))
    if variant == "compact":
        phi = _neumann(div - div.mean(), n, h)
        edge = 0
    else:
        phi, edge = torch.empty_like(div), 1
        for a in range(8):
            cl = (slice(a >> 2 & 1, None, 2), slice(a >> 1 & 1, None, 2), slice(a & 1, None, 2))
            b = div[cl]
            phi[cl] = _neumann(b - b.mean(), [m // 2 for m in n], [2 * v for v in h])
    return torch.stack([B[d] - _central(phi, 2 - d, h[d], edge) for d in range(3)])


def _psi_direct(n, lo, hi, U, geom):
    """psi of lap u + 2 pi U / (1 + u) = 0, u = psi - 1, Robin outer condition: Newton's method, each step a block
    tridiagonal solve along the longer dimension of the flux-form operator."""
    n0, n1 = n
    h0, h1 = (hi[0] - lo[0]) / n0, (hi[1] - lo[1]) / n1
    x, y = _centres(n, lo, hi)
    xp, xm = x + 0.5 * h0, x - 0.5 * h0
    p = 2 if geom == "sph" else 1
    # operator as five diagonals on the (n1, n0) grid, ghosts folded into the centre
    one = np.ones((n1, n0))
    cE, cW = one * (xp / x) ** p / h0 ** 2, one * (xm / x) ** p / h0 ** 2
    if geom == "sph":
        s = np.sin(y)
        sf = np.sin(lo[1] + np.arange(n1 + 1) * h1)
        sf[0] = sf[-1] = 0.0
        cN, cS = ((sf[1:] / s)[:, None] / h1 ** 2) / x ** 2, ((sf[:-1] / s)[:, None] / h1 ** 2) / x ** 2
    else:
        cN, cS = one / h1 ** 2, one / h1 ** 2
    cC = -(cE + cW + cN + cS)
    cW[:, 0] = 0.0
    cC[:, 0] = -(cE + cN + cS)[:, 0]
    if geom == "sph":
        cC[:, -1] += cE[:, -1] * x[-1] / (x[-1] + h0)
    else:
        dist = lambda a, b: np.sqrt(a * a + b * b)
        cC[:, -1] += cE[:, -1] * dist(x[-1], y) / dist(x[-1] + h0, y)
        cC[-1] += cN[-1] * dist(x, y[-1]) / dist(x, y[-1] + h1)
        cC[0] += cS[0] * dist(x, y[0]) / dist(x, y[0] - h1)
        cN[-1] = 0.0
        cS[0] = 0.0
    cE[:, -1] = 0.0
    if n0 < n1:  # march along the longer dimension
        lower, upper, left, right, centre, src = cS, cN, cW, cE, cC, U
    else:
        lower, upper, left, right, centre, src = cW.T, cE.T, cS.T, cN.T, cC.T, U.T
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    lower, upper, left, right, centre, src = (t(a) for a in (lower, upper, left, right, centre, src))
    m, b = src.shape

    def apply(u):
        r = centre * u
        r[1:] += lower[1:] * u[:-1]
        r[:-1] += upper[:-1] * u[1:]
        r[:, 1:] += left[:, 1:] * u[:, :-1]
        r[:, :-1] += right[:, :-1] * u[:, 1:]
        return r

    u = torch.zeros_like(src)
    for _ in range(8):
        F = apply(u) + 2 * PI * src / (1 + u)
        diag = centre - 2 * PI * src / (1 + u) ** 2
        E, g = [], []
        for i in range(m):
            T = torch.diag(diag[i]) + torch.diag(left[i, 1:], -1) + torch.diag(right[i, :-1], 1)
            rhs = -F[i]
            if i:
                T = T - lower[i][:, None] * E[-1]
                rhs = rhs - lower[i] * g[-1]
            sol = torch.linalg.solve(T, torch.cat([torch.diag(upper[i]), rhs[:, None]], 1))
            E.append(sol[:, :b])
            g.append(sol[:, b])
        d = [None] * m
        d[-1] = g[-1]
        for i in range(m - 2, -1, -1):
            d[i] = g[i] - E[i] @ d[i + 1]
        step = torch.stack(d)
        u = u + step
        if float(step.abs().max()) < 1e-15:
            break
    u = u if n0 < n1 else u.T
    return (1.0 + u).contiguous()
