"""What a user of this library runs, as cases that can be timed.

Every case is a call (or the few calls that belong together) of the public
binding `paper_1405_6456_gb300.ofdft`, on FCC aluminium-like clusters of
cx x cy x cz cells with seeded displacements of 0.1 bohr, Z = 3, sigma = 1 bohr:
the clusters of `workloads.py`, of the tests and of bench.py.  The grid is the
library's box rule at the case's spacing, vacuum and rounding (rounding 1 gives
odd extents).  `exact` restates the method in 64 bits with torch alone.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1405_6456_gb300 import ofdft as F
from paper_1405_6456_gb300 import workloads as W

DEV = "cuda:0"
A_LAT, Z_ION, SIGMA, RCUT = 7.6, 3.0, 1.0, 7.0   # bohr, charge, Gaussian width, ball radius (library defaults)
GUESS_SIGMA, GUESS_CUT, LAMBDA = 2.0, 8.0, 0.2

_context = None


def _ctx():
    """One context for the whole program, as a user keeps it."""
    global _context
    if _context is None:
        _context = F.Context(0)
    return _context


# ------------------------------------------------------------------ the cases --
def _case(name, kind, prec, cells, h, order, vacuum, round_to=16, **more):
    return {"name": name, "kind": kind, "prec": prec, "cx": cells[0], "cy": cells[1], "cz": cells[2], "h": h,
            "order": order, "vacuum": vacuum, "round_to": round_to, **more}


def listed():
    return [
        # one application of L_h to a field a caller already has; the 192^3 field of the 2457-atom cluster in FP32
        _case("stencil_f32_192", "stencil", "mixed", (8, 8, 8), 0.45, 12, 10.0),
        # the same on a grid the caller's own box rule left with odd extents (rows that are not whole vectors), FP64
        _case("stencil_f64_odd", "stencil", "fp64", (4, 3, 5), 0.5, 8, 9.0, 1),
        # the smallest Poisson solve in use: the 13/14-atom clusters' 32..48^3 grids, where launches count
        _case("poisson_f64_small", "poisson", "fp64", (1, 1, 1), 0.6, 12, 8.0, tol=1e-10, source="ub"),
        # the plain FP64 method's Poisson solve at 666 atoms, 128^3
        _case("poisson_f64_128", "poisson", "fp64", (5, 5, 5), 0.5, 12, 10.0, tol=1e-10, source="ub"),
        # mixed precision on an odd, elongated box (a rod), lower order, an explicit density
        _case("poisson_f32_odd", "poisson", "mixed", (2, 3, 6), 0.5, 8, 8.0, 1, tol=1e-8, source="rho"),
        # the Poisson solve of the benchmark's 2457-atom cluster, 192^3, from phi = 0
        _case("poisson_f32_192", "poisson", "mixed", (8, 8, 8), 0.45, 12, 10.0, tol=1e-8, source="ub"),
        # the method's unit of work: L and its gradient at a line search's trial point, phi warm-started; FP64
        _case("evaluate_f64_80", "evaluate", "fp64", (3, 3, 3), 0.5, 12, 8.0, tol=1e-10),
        # the same in MIXED at the benchmark's size
        _case("evaluate_f32_192", "evaluate", "mixed", (8, 8, 8), 0.45, 12, 10.0, tol=1e-8),
        # what every new geometry pays first: pseudocharge with its self energy, and the starting guess
        _case("setup_f64_128", "setup", "fp64", (5, 5, 5), 0.5, 12, 10.0),
        # forces on the nuclei of a converged potential (geometry steps), paper form
        _case("forces_f64_112", "forces", "fp64", (4, 4, 4), 0.45, 12, 8.0, variant=F.FORCE_PAPER),
        # a whole ground state, energy only (as the binding-energy series computes it), MIXED, 666 atoms
        _case("solve_f32_128", "solve", "mixed", (5, 5, 5), 0.5, 12, 10.0),
        # six uneven clusters through the batch engine, MIXED (screening: their energies)
        _case("batch_f32", "batch", "mixed", (1, 2, 3), 0.5, 12, 8.0, count=6),
    ]


_KINDS = ("stencil", "stencil", "poisson", "poisson", "poisson", "evaluate", "evaluate", "evaluate", "setup", "forces",
          "solve", "batch")


def draw(rng):
    """One more case: a kind in the proportions of use, cells, spacing, order,
    vacuum and rounding over the ranges the listed ones stand for."""
    kind = rng.choice(_KINDS)
    prec = rng.choice(("mixed", "fp64"))
    h = rng.choice((0.45, 0.5, 0.55, 0.6, 0.8))
    order = rng.choice((6, 8, 10, 12, 12, 12))
    vacuum = rng.choice((8.0, 9.0, 10.0))
    round_to = rng.choice((1, 2, 16, 16))
    if kind in ("solve", "batch"):
        prec, h = "mixed", rng.choice((0.5, 0.6))
        order = rng.choice((8, 12))
    most = {"solve": 4, "batch": 2, "setup": 5, "forces": 5}.get(kind, 8 if prec == "mixed" else 5)
    # log-uniform numbers of cells, the three axes apart; whole clusters are mostly cubes
    cells = [min(most, int(math.exp(rng.uniform(0.0, math.log(most + 1.0))))) for _ in range(3)]
    if kind not in ("stencil", "poisson") and rng.random() < 0.6:
        cells = [max(cells)] * 3
    c = {"kind": kind, "prec": prec, "cx": cells[0], "cy": cells[1], "cz": cells[2], "h": h, "order": order,
         "vacuum": vacuum, "round_to": round_to}
    if kind in ("poisson", "evaluate"):
        c["tol"] = 1e-8 if prec == "mixed" else 1e-10
    if kind == "poisson":
        c["source"] = rng.choice(("rho", "ub"))
    if kind == "forces":
        c["variant"] = F.FORCE_PAPER
    if kind == "batch":
        c["cx"], c["cy"], c["cz"] = 1, 1, 2
        c["count"] = rng.randint(2, 6)
    return c


# ------------------------------------------------------------------- geometry --
def _sites(cx, cy, cz):
    """FCC sites of cx x cy x cz cells, centred (fcc_cube_sites for a cube)."""
    i, j, k = np.meshgrid(np.arange(2 * cx + 1), np.arange(2 * cy + 1), np.arange(2 * cz + 1), indexing="ij")
    keep = ((i + j + k) % 2) == 0
    pts = np.stack([i[keep], j[keep], k[keep]], axis=1) * (A_LAT / 2.0)
    return pts - 0.5 * A_LAT * np.array([cx, cy, cz])


def _atoms(c, seed):
    R = W.displaced(_sites(c["cx"], c["cy"], c["cz"]), 0.1, seed)
    return R, np.full(R.shape[0], Z_ION)


def _grid(c):
    """The box rule for the undisplaced sites, so that a case's sizes do not depend on the seed."""
    return F.ofdft_grid_for_atoms(_sites(c["cx"], c["cy"], c["cz"]), c["h"], c["vacuum"], c["round_to"])


def _dtype(c):
    return torch.float64 if c["prec"] == "fp64" else torch.float32


def _prec(c):
    return F.PREC_FP64 if c["prec"] == "fp64" else F.PREC_MIXED


def _axes(g):
    """Node coordinates along x, y, z (cell-centred)."""
    return [torch.as_tensor([g.origin[d] + (i + 0.5) * g.h for i in range(g.n[d])], dtype=torch.float64, device=DEV)
            for d in range(3)]


def _weights(n, h):
    """(w_0, [w_1 .. w_n]) of the order-2n second-derivative stencil."""
    w0 = -sum(1.0 / q**2 for q in range(1, n + 1)) / h**2
    w = [2.0 * (-1) ** (p + 1) / (h**2 * p**2) * math.factorial(n) ** 2 / (math.factorial(n - p) * math.factorial(n + p))
         for p in range(1, n + 1)]
    return w0, w


def _laplacian(f, n, h):
    """L_h f in 64 bits, zero outside the grid; f[z, y, x] (leading axes are batched)."""
    w0, w = _weights(n, h)
    out = (6.0 * w0) * f
    for p in range(1, n + 1):
        for ax in (-3, -2, -1):
            if f.shape[ax] > p:
                m = f.shape[ax] - p
                out.narrow(ax, 0, m).add_(f.narrow(ax, p, m), alpha=w[p - 1])
                out.narrow(ax, p, m).add_(f.narrow(ax, 0, m), alpha=w[p - 1])
    return out


def _solve_poisson(rho, n, h):
    """phi of (-L_h) phi = 4 pi rho in 64 bits: the three axes' matrices diagonalised."""
    w0, w = _weights(n, h)
    f = (4.0 * math.pi) * rho.double()
    vals, vecs = [], []
    for m in (f.shape[2], f.shape[1], f.shape[0]):
        T = torch.zeros(m, m, dtype=torch.float64)
        T.diagonal().fill_(-2.0 * w0)
        for p in range(1, min(n, m - 1) + 1):
            T.diagonal(p).fill_(-w[p - 1])
            T.diagonal(-p).fill_(-w[p - 1])
        lam, Q = torch.linalg.eigh(T)
        vals.append(lam.to(DEV))
        vecs.append(Q.to(DEV))
    qx, qy, qz = vecs

    def apply(f, a, b, c):  # f[z, y, x] times a, b, c along x, y, z
        f = torch.matmul(f, a)
        f = torch.matmul(b.T, f)
        return torch.matmul(c.T, f.reshape(f.shape[0], -1)).reshape(f.shape)

    f = apply(f, qx, qy, qz)
    f /= vals[2][:, None, None] + vals[1][None, :, None] + vals[0][None, None, :]
    return apply(f, qx.T, qy.T, qz.T)


def _boxes(g, R, reach):
    """Index ranges of the nodes that can lie within `reach` of each atom, unclipped: (first index (M, 3), length)."""
    half = int(math.ceil(reach / g.h)) + 1
    o = np.array([g.origin[d] for d in range(3)])
    lo = np.floor((R - o) / g.h - 0.5).astype(np.int64) - half + 1
    return lo, 2 * half + 1


def _box_offsets(g, R, lo, m):
    """Offsets node - atom along the three axes of every box, (M, m) each."""
    i = np.arange(m)
    return [torch.as_tensor((g.origin[d] + (lo[:, d:d + 1] + i + 0.5) * g.h) - R[:, d:d + 1], device=DEV)
            for d in range(3)]


def _radius(off):
    x, y, z = off
    return torch.sqrt((x * x)[:, None, None, :] + (y * y)[:, None, :, None] + (z * z)[:, :, None, None])


def _v_nucleus(r):
    return torch.where(r < 1e-12, torch.full_like(r, -2.0 * Z_ION / (SIGMA * math.sqrt(math.pi))),
                       -Z_ION * torch.erf(r / SIGMA) / r.clamp_min(1e-300))


def _add_boxes(out, g, lo, vals):
    """out[z, y, x] += the boxes' in-grid parts."""
    n, m = g.n, vals.shape[-1]
    for a in range(vals.shape[0]):
        l = [int(v) for v in lo[a]]
        s = [(max(0, -l[d]), min(m, n[d] - l[d])) for d in range(3)]
        if any(e <= b for b, e in s):
            continue
        (xb, xe), (yb, ye), (zb, ze) = s
        out[l[2] + zb:l[2] + ze, l[1] + yb:l[1] + ye, l[0] + xb:l[0] + xe] += vals[a, zb:ze, yb:ye, xb:xe]


def _charge_boxes(g, R, n):
    """Per chunk of atoms: (slice, box starts, b_J, V_J on the ball's box, b_J with a halo of n)."""
    for a0 in range(0, R.shape[0], 64):
        Rc = R[a0:a0 + 64]
        lo, m = _boxes(g, Rc, RCUT)
        lo2, m2 = lo - 2 * n, m + 4 * n
        V = _v_nucleus(_radius(_box_offsets(g, Rc, lo2, m2)))
        b = (-1.0 / (4.0 * math.pi)) * _laplacian(V, n, g.h)[:, n:-n, n:-n, n:-n]
        r = _radius(_box_offsets(g, Rc, lo - n, m + 2 * n))
        b = torch.where(r < RCUT, b, torch.zeros_like(b))
        inner = slice(n, -n)
        yield slice(a0, a0 + Rc.shape[0]), lo, b[:, inner, inner, inner], V[:, 2 * n:-2 * n, 2 * n:-2 * n,
                                                                            2 * n:-2 * n], b


def _inside(g, lo, m):
    """Which box nodes lie in the grid, (atoms, m, m, m)."""
    i = torch.arange(m, device=DEV)
    ok = []
    for d in range(3):
        k = torch.as_tensor(lo[:, d:d + 1], device=DEV) + i
        ok.append((k >= 0) & (k < g.n[d]))
    return ok[0][:, None, None, :] & ok[1][:, None, :, None] & ok[2][:, :, None, None]


def _pseudocharge(g, R, n):
    """b on the grid and the self energy, in 64 bits."""
    b = torch.zeros(g.shape, dtype=torch.float64, device=DEV)
    es = 0.0
    for _, lo, bj, vj, _ in _charge_boxes(g, R, n):
        _add_boxes(b, g, lo, bj)
        es += float((bj * vj * _inside(g, lo, bj.shape[-1])).sum())
    return b, 0.5 * g.h**3 * es


def _guess(g, R, N):
    """The starting guess: root of the superposed, cut atomic Gaussians, normalised to N."""
    rho = torch.zeros(g.shape, dtype=torch.float64, device=DEV)
    norm = (2.0 * math.pi * GUESS_SIGMA**2) ** -1.5
    for a0 in range(0, R.shape[0], 64):
        Rc = R[a0:a0 + 64]
        lo, m = _boxes(g, Rc, GUESS_CUT)
        x, y, z = _box_offsets(g, Rc, lo, m)
        r2 = (x * x)[:, None, None, :] + (y * y)[:, None, :, None] + (z * z)[:, :, None, None]
        v = Z_ION * norm * torch.exp(-r2 / (2.0 * GUESS_SIGMA**2))
        _add_boxes(rho, g, lo, torch.where(r2 < GUESS_CUT**2, v, torch.zeros_like(v)))
    u = torch.sqrt(rho)
    return u * math.sqrt(N / (g.h**3 * float((u * u).sum())))


def _noise(g, gen, modes=4):
    """A smooth random field of order one: a few random cosines along each axis."""
    out = torch.zeros(g.shape, dtype=torch.float64, device=DEV)
    for _ in range(modes):
        k = torch.rand(3, generator=gen, dtype=torch.float64) * 6.0 + 0.5
        ph = torch.rand(3, generator=gen, dtype=torch.float64) * 2.0 * math.pi
        ax = [torch.cos(float(k[d]) * torch.linspace(0, 1, g.n[d], dtype=torch.float64, device=DEV) + float(ph[d]))
              for d in range(3)]
        out += ax[2][:, None, None] * ax[1][None, :, None] * ax[0][None, None, :]
    return out / math.sqrt(modes)


# -------------------------------------------------------------------- prepare --
def _fields(c, seed):
    """Geometry, grid and, in 64 bits, the fields the case's call takes."""
    R, Z = _atoms(c, seed)
    g = _grid(c)
    n, kind = c["order"] // 2, c["kind"]
    f = {"R": R, "Z": Z, "g": g}
    if kind in ("setup", "solve", "batch"):
        return f
    gen = torch.Generator().manual_seed(seed)
    u = _guess(g, R, float(Z.sum()))
    u = (u * (1.0 + 0.05 * _noise(g, gen))).abs()
    if kind == "stencil":
        f["f"] = u
        return f
    f["u"] = u
    f["b"], f["E_self"] = _pseudocharge(g, R, n)
    if kind == "poisson":
        f["phi"] = torch.zeros_like(u)
    elif kind == "forces":
        f["phi"] = _solve_poisson(u * u + f["b"], n, g.h)
    elif kind == "evaluate":
        # a trial point u + d of a line search, phi still that of its origin u
        f["phi"] = _solve_poisson(u * u + f["b"], n, g.h)
        f["d"] = 0.02 * u * (1.0 + 0.5 * _noise(g, gen))
        f["s_old"] = 0.02 * u * (1.0 + 0.5 * _noise(g, gen))
        f["u"] = (u + f["d"]).abs()
    return f


def prepare(case, seed):
    f = _fields(case, seed)
    dt, kind = _dtype(case), case["kind"]
    st = {"case": case, "ctx": _ctx(), "g": f["g"], "R": f["R"], "Z": f["Z"], "N": float(f["Z"].sum())}
    new = lambda: torch.empty(f["g"].shape, dtype=dt, device=DEV)  # noqa: E731
    for k in ("f", "u", "b", "phi", "d", "s_old"):
        if k in f:
            st[k] = f[k].to(dt)
    if kind == "stencil":
        st["out"] = new()
    elif kind == "poisson":
        if case["source"] == "rho":
            st["rho"] = (f["u"] * f["u"] + f["b"]).to(dt)
        st["out"] = new()
    elif kind == "evaluate":
        st["E_self"] = f["E_self"]
        st["params"] = F.default_params(fd_order=case["order"], precision=_prec(case), tol_poisson=case["tol"])
        st["out"], st["G"], st["s"] = new(), new(), new()
    elif kind == "setup":
        st["b"], st["u"] = new(), new()
    elif kind in ("solve", "batch"):
        st["params"] = F.default_params(fd_order=case["order"], precision=_prec(case), vacuum=case["vacuum"],
                                        round_to=case["round_to"])
        if kind == "batch":
            rng = np.random.Generator(np.random.PCG64(case["count"]))
            cells = [tuple(int(v) for v in rng.choice([case["cx"], case["cy"], case["cz"]], size=1)) * 3
                     for _ in range(case["count"])]
            cells[0] = (case["cz"],) * 3  # the largest is always among them
            st["many"] = []
            for i, (m, _, _) in enumerate(cells):
                R = W.displaced(_sites(m, m, m), 0.1, seed + 1000 * (i + 1))
                st["many"].append((R, np.full(R.shape[0], Z_ION), F.ofdft_grid_for_atoms(
                    _sites(m, m, m), case["h"], case["vacuum"], case["round_to"])))
            st["batch"] = F.Batch(_ctx(), _prec(case), 16 << 30)
    return st


# ------------------------------------------------------------------------ run --
_ENERGIES = ("L", "E", "E_tf", "E_vw", "E_xc", "E_es", "gd", "gs_old", "gnorm2", "rs", "rs_pc")


def run(st):
    c, ctx, g, order = st["case"], st["ctx"], st["g"], st["case"]["order"]
    kind = c["kind"]
    if kind == "stencil":
        ctx.stencil(g, order, st["f"], st["out"])
        return st["out"]
    if kind == "poisson":
        st["out"].copy_(st["phi"])  # the incoming guess
        if c["source"] == "rho":
            ctx.poisson(g, order, st["out"], rho=st["rho"], tol=c["tol"])
        else:
            ctx.poisson(g, order, st["out"], u=st["u"], b=st["b"], tol=c["tol"])
        return st["out"]
    if kind == "evaluate":
        st["out"].copy_(st["phi"])
        e = ctx.energy_grad(g, st["params"], st["u"], st["b"], st["out"], st["E_self"], -0.2, 0.1, st["N"],
                            grad=st["G"], s=st["s"], d=st["d"], s_old=st["s_old"])
        return {"phi": st["out"], "grad": st["G"], "s": st["s"], **{k: getattr(e, k) for k in _ENERGIES}}
    if kind == "setup":
        es = ctx.pseudocharge(g, order, st["R"], st["Z"], st["b"], sigma=SIGMA, rc=RCUT)
        ctx.initial_guess(g, st["R"], st["Z"], st["u"], guess_sigma=GUESS_SIGMA, guess_cut=GUESS_CUT)
        return {"b": st["b"], "u": st["u"], "E_self": es}
    if kind == "forces":
        return ctx.forces(g, order, st["R"], st["Z"], st["phi"], sigma=SIGMA, rc=RCUT, variant=c["variant"])
    if kind == "solve":
        E, _, stats = ctx.solve(st["R"], st["Z"], c["h"], st["params"], grid=g, want_forces=False)
        return {"E": E, "converged": bool(stats.converged)}
    ids = [st["batch"].submit(R, Z, c["h"], st["params"], grid=gg) for R, Z, gg in st["many"]]
    st["batch"].run()
    return {"E": [st["batch"].poll(i)[0] for i in ids]}


# ----------------------------------------------------------------------- work --
def work(case):
    es = 8 if case["prec"] == "fp64" else 4
    kind, n = case["kind"], case["order"] // 2
    if kind == "batch":
        rng = np.random.Generator(np.random.PCG64(case["count"]))
        ms = [int(rng.choice([case["cx"], case["cy"], case["cz"]], size=1)[0]) for _ in range(case["count"])]
        ms[0] = case["cz"]
        all_sites = [_sites(m, m, m) for m in ms]
    else:
        all_sites = [_sites(case["cx"], case["cy"], case["cz"])]
    nodes = [F.ofdft_grid_for_atoms(s, case["h"], case["vacuum"], case["round_to"]).size for s in all_sites]
    G, M = float(sum(nodes)), float(sum(len(s) for s in all_sites))
    lap = 2.0 * (6 * n + 1)                        # one L_h at one node
    ball = 4.0 / 3.0 * math.pi * (RCUT / case["h"]) ** 3  # nodes of one atom's ball
    setup = M * ball * (lap + 40.0) + M * 4.0 / 3.0 * math.pi * (GUESS_CUT / case["h"]) ** 3 * 20.0
    if kind == "stencil":
        return {"bytes": 2.0 * G * es, "flops": G * lap}
    if kind == "poisson":  # u and b (or rho) and phi in, phi out; the residual before and after
        return {"bytes": G * es * (3.0 if case["source"] == "rho" else 4.0), "flops": G * 2.0 * (lap + 6.0)}
    if kind == "evaluate":  # u, b, phi, d, s_old in; phi, grad, s out; the Poisson residuals and the functional
        return {"bytes": G * es * 8.0, "flops": G * (3.0 * lap + 80.0)}
    if kind == "setup":
        return {"bytes": 2.0 * G * es, "flops": setup}
    if kind == "forces":
        return {"bytes": G * es, "flops": M * ball * (lap + 40.0 + 6.0 * 2.0 * n)}
    # a ground state: the set-up and, at the least, the evaluations at its start and its end
    return {"bytes": 2.0 * G * es * 8.0, "flops": setup + 2.0 * G * (3.0 * lap + 80.0)}


# ---------------------------------------------------------------------- exact --
def _xc(rho):
    """eps_xc and V_xc of the Perdew-Zunger form with the paper's constants; zero below the density floor."""
    r13 = rho.clamp_min(1e-30) ** (1.0 / 3.0)
    c = (3.0 / math.pi) ** (1.0 / 3.0)
    rs = (3.0 / (4.0 * math.pi)) ** (1.0 / 3.0) / r13
    g1, b1, b2 = -0.1423, 1.0529, 0.3334
    A, B, C, D = 0.0311, -0.048, 0.002, -0.0116
    q, den = torch.sqrt(rs), 1.0 + b1 * torch.sqrt(rs) + b2 * rs
    lo_e, lo_v = g1 / den, g1 * (1.0 + 7.0 / 6.0 * b1 * q + 4.0 / 3.0 * b2 * rs) / den**2
    ln = torch.log(rs)
    hi_e = A * ln + B + C * rs * ln + D * rs
    hi_v = A * ln + (B - A / 3.0) + 2.0 / 3.0 * C * rs * ln + (2.0 * D - C) / 3.0 * rs
    on = rho >= 1e-30
    zero = torch.zeros_like(rho)
    eps = torch.where(on, -0.75 * c * r13 + torch.where(rs >= 1.0, lo_e, hi_e), zero)
    v = torch.where(on, -c * r13 + torch.where(rs >= 1.0, lo_v, hi_v), zero)
    return eps, v


def _exact_evaluate(case, st):
    n, h = case["order"] // 2, st["g"].h
    h3, N, eta, mu = h**3, st["N"], -0.2, 0.1
    u, b, d, s_old = (st[k].double() for k in ("u", "b", "d", "s_old"))
    rho = u * u
    phi = _solve_poisson(rho + b, n, h)
    lap = _laplacian(u, n, h)
    cf = 0.3 * (3.0 * math.pi**2) ** (2.0 / 3.0)
    u43 = u.abs() ** (4.0 / 3.0)
    eps, vxc = _xc(rho)
    E_tf, E_vw, E_xc = (h3 * float(t.sum()) for t in (cf * u43 * rho, -0.5 * LAMBDA * u * lap, eps * rho))
    lphi = _laplacian(phi, n, h)
    E_es = h3 * float((phi * lphi / (8.0 * math.pi) + (rho + b) * phi).sum()) - st["E_self"]
    C = h3 * float(rho.sum()) - N
    E = E_tf + E_vw + E_xc + E_es
    mult = -eta + C / mu
    vk = 5.0 / 3.0 * cf * u43
    G = -LAMBDA * lap + 2.0 * (vk + vxc + phi) * u + 2.0 * mult * u
    kin = -6.0 * LAMBDA * _weights(n, h)[0] + 14.0 / 3.0 * vk
    diag = torch.maximum(kin + 2.0 * (vxc + phi + mult), 0.25 * kin).clamp_min(1e-10)
    s, w = -G / diag, u / diag
    cpen = 4.0 * h3 / mu
    us = float((u * s).sum())
    gamma = cpen * us / (1.0 + cpen * float((u * w).sum()))
    rs = h3 * float((G * -s).sum())
    return {"phi": phi, "grad": G, "s": s - gamma * w, "L": E - eta * C + 0.5 * C * C / mu, "E": E, "E_tf": E_tf,
            "E_vw": E_vw, "E_xc": E_xc, "E_es": E_es, "gd": h3 * float((G * d).sum()),
            "gs_old": h3 * float((G * s_old).sum()), "gnorm2": h3 * float((G * G).sum()), "rs": rs,
            "rs_pc": rs - h3 * gamma * us}


def _exact_forces(case, st):
    n, g = case["order"] // 2, st["g"]
    phi = st["phi"].double()
    w = [(-1) ** (p + 1) * math.factorial(n) ** 2 / (g.h * p * math.factorial(n - p) * math.factorial(n + p))
         for p in range(1, n + 1)]
    out = np.zeros((st["R"].shape[0], 3))
    for at, lo, _, vj, bh in _charge_boxes(g, st["R"], n):
        m = vj.shape[-1]
        pj = torch.zeros_like(vj)
        for a in range(vj.shape[0]):
            l = [int(v) for v in lo[a]]
            (xb, xe), (yb, ye), (zb, ze) = [(max(0, -l[k]), min(m, g.n[k] - l[k])) for k in range(3)]
            pj[a, zb:ze, yb:ye, xb:xe] = phi[l[2] + zb:l[2] + ze, l[1] + yb:l[1] + ye, l[0] + xb:l[0] + xe]
        r = _radius(_box_offsets(g, st["R"][at], lo, m))
        pv = torch.where((r < RCUT) & _inside(g, lo, m), pj - vj, torch.zeros_like(vj))
        for k, ax in enumerate((3, 2, 1)):
            grad = torch.zeros_like(vj)
            for p in range(1, n + 1):
                idx = [slice(None)] + [slice(n, n + m)] * 3
                up, dn = list(idx), list(idx)
                up[ax], dn[ax] = slice(n + p, n + p + m), slice(n - p, n - p + m)
                grad += w[p - 1] * (bh[tuple(up)] - bh[tuple(dn)])
            out[at, k] = g.h**3 * (grad * pv).sum(dim=(1, 2, 3)).cpu().numpy()
    return out


def exact(case, seed):
    kind, n = case["kind"], case["order"] // 2
    if kind in ("solve", "batch"):
        return None  # a whole minimisation in 64 bits takes minutes
    st = prepare(case, seed)
    h = st["g"].h
    if kind == "stencil":
        return _laplacian(st["f"].double(), n, h)
    if kind == "poisson":
        rho = st["rho"].double() if case["source"] == "rho" else st["u"].double() ** 2 + st["b"].double()
        return _solve_poisson(rho, n, h)
    if kind == "evaluate":
        return _exact_evaluate(case, st)
    if kind == "setup":
        b, es = _pseudocharge(st["g"], st["R"], n)
        return {"b": b, "u": _guess(st["g"], st["R"], st["N"]), "E_self": es}
    return _exact_forces(case, st)
