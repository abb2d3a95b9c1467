"""Fast diagonalisation as the Poisson CG's preconditioner, through the C ABI, at
the sizes where its panels, tiles and halves have edges.

The right-hand side is the discrete operator applied to a known field (the
oracle's stencil), so the solve must return that field.  Tolerance, from
||phi - phi*|| <= ||A^-1|| ||r|| with ||r|| <= tol ||4 pi rho||: relative to
||phi*|| at most tol times the operator's condition number, of which the largest
and smallest eigenvalues are bounded by the symbol: lambda_max <= 12 / h^2 sum_p
|w_p h^2| and lambda_min >= 3 (pi / (n_max + 1))^2 / h^2 / 2; FP32 results add
their rounding (2^-24 a value, doubled).
"""
import os

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
from paper_1405_6456_gb300 import build as B
from paper_1405_6456_gb300 import ofdft as F

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _context(**env):
    old = {k: os.environ.get(k) for k in env}
    os.environ.update({k: str(v) for k, v in env.items()})
    try:
        return F.Context(0)
    finally:
        for k, v in old.items():
            if v is None:
                del os.environ[k]
            else:
                os.environ[k] = v


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.build()
    c = F.Context(0)
    yield c
    c.close()


# the shortest axis; odd halves, rows that are no whole vectors; one node past a
# tile; two tiles a warp (more than 256 nodes) on each axis in turn; the longest
SIZES = [((32, 32, 32), 12), ((33, 35, 34), 12), ((47, 40, 39), 2), ((64, 97, 36), 8), ((130, 33, 66), 6),
         ((257, 32, 33), 12), ((32, 300, 34), 10), ((36, 32, 512), 12), ((512, 32, 32), 4)]


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("dims,order", SIZES)
def test_poisson_returns_the_known_field(ctx, dims, order, dtype):
    g = F.make_grid(*dims, 0.5)
    og = O.make_grid(*dims, 0.5, (0.0, 0.0, 0.0))
    phi_m = np.random.default_rng(sum(dims)).standard_normal(g.shape)
    rho = -O.laplacian(og, order // 2, phi_m) / (4.0 * np.pi)
    if dtype == torch.float32:
        rho = rho.astype(np.float32)
    tol = 1e-10 if dtype == torch.float64 else 1e-8
    phi = torch.zeros(g.shape, dtype=dtype, device=DEV)
    ctx.reset_counters()
    st = ctx.poisson(g, order, phi, rho=torch.as_tensor(rho, device=DEV), tol=tol)
    cnt = ctx.counters()
    assert st.rel_residual <= tol
    n = cnt.kind_launches[F.K_MG]  # five passes a step or correction, some launched ahead
    assert n % 5 == 0 and 5 * st.iterations <= n <= 5 * (st.iterations + 1)
    assert st.iterations <= 6  # V-cycles: 17 to 35
    w = np.abs(O.lap_weights(order // 2, 1.0))
    lam_max, lam_min = 12.0 * w[1:].sum(), 1.5 * (np.pi / (max(dims) + 1)) ** 2
    cond = lam_max / lam_min
    bound = tol * cond
    if dtype == torch.float32:
        # rho itself is rounded to FP32 (2^-25 a value), which A^-1 carries to phi
        bound += 2.0**-25 * cond + 2.0**-23
    err = np.linalg.norm(phi.double().cpu().numpy() - phi_m) / np.linalg.norm(phi_m)
    assert err <= bound, (err, bound)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_unaligned_fields_and_the_vcycle_agree(ctx, dtype):
    """Fields that start off a 16-byte boundary take the element-wise rows of the x
    passes; the V-cycle (OFDFT_FD=0) reaches the same potential."""
    dims, order = (48, 40, 36), 12
    g = F.make_grid(*dims, 0.5)
    rho = np.random.default_rng(4).standard_normal(g.shape)
    tol = 1e-10 if dtype == torch.float64 else 1e-9
    sols = []
    cv = _context(OFDFT_FD=0)
    for c, off in ((ctx, 0), (ctx, 1), (cv, 0)):
        buf = torch.zeros(2, g.size + 1, dtype=dtype, device=DEV)
        phi, r = (buf[k, off:off + g.size].view(g.shape) for k in (0, 1))
        r.copy_(torch.as_tensor(rho))
        st = c.poisson(g, order, phi, rho=r, tol=tol)
        assert st.rel_residual <= tol
        sols.append(phi.double().cpu().numpy())
    cv.close()
    # each is within tol * cond of the solution (cond <= 27 / 6.5e-3 at n = 48), FP32 ones with their rounding
    bound = 2.0 * (tol * 4.2e3 + (0.0 if dtype == torch.float64 else 2.0**-23))
    for s in sols[1:]:
        assert np.linalg.norm(s - sols[0]) <= bound * np.linalg.norm(sols[0])


def test_short_axes_keep_the_vcycle(ctx):
    """One axis below 32 nodes: the multigrid launches of one iteration are not the
    five passes."""
    g = F.make_grid(31, 40, 40, 0.5)
    rho = torch.as_tensor(np.random.default_rng(4).standard_normal(g.shape), device=DEV)
    phi = torch.zeros(g.shape, dtype=torch.float64, device=DEV)
    ctx.reset_counters()
    st = ctx.poisson(g, 12, phi, rho=rho, tol=1e-10)
    assert st.iterations > 6
    assert ctx.counters().kind_launches[F.K_MG] > 5 * st.iterations


@pytest.mark.parametrize("prec", [F.PREC_FP64, F.PREC_MIXED])
def test_batched_passes_do_not_depend_on_the_mix(ctx, prec):
    """Grids of one and of two output tiles a warp in one batch (one axis over 128
    nodes), beside one that keeps the V-cycle: each result is the same alone, bit for
    bit, and the single solve's within the solver's tolerance (E is second order in
    what tol_inner leaves: 1e-8 Ha/atom, a tenth of the bound)."""
    from paper_1405_6456_gb300 import workloads as W
    c = W.tiny_cluster("dimer", h=0.6, fd_order=8)
    p = F.default_params(fd_order=8, precision=prec, tol_E=1e-7, tol_inner=1e-8)
    grids = []
    for n in ((44, 34, 36), (140, 33, 34), (44, 30, 32)):
        grids.append(F.make_grid(*n, 0.6, tuple(-0.3 * k for k in n)))
    alone = []
    for g in grids:
        bt = F.Batch(ctx, prec, 1 << 32)
        rid = bt.submit(c.R, c.Z, c.h, p, grid=g)
        bt.run()
        alone.append(bt.poll(rid))
        bt.close()
    bt = F.Batch(ctx, prec, 1 << 32)
    ids = [bt.submit(c.R, c.Z, c.h, p, grid=g) for g in grids]
    bt.run()
    for g, rid, (Ea, Fa, _) in zip(grids, ids, alone):
        E, Fv, st = bt.poll(rid)
        assert st.converged and E == Ea and np.array_equal(Fv, Fa)
        E1, _, _ = ctx.solve(c.R, c.Z, c.h, p, grid=g)
        assert abs(E - E1) / c.M <= 1e-7
    bt.close()


@pytest.mark.parametrize("dims", [(45, 35, 37), (44, 36, 38)])
def test_mixed_ground_state_with_odd_and_even_node_counts(ctx, dims):
    """The passes that prepare the potential and add a correction take two nodes a
    lane only where the node count is even: a ground state either way is the V-cycle
    form's (tolerance as in the batch test above: a tenth of it is E's own error)."""
    from paper_1405_6456_gb300 import workloads as W
    c = W.tiny_cluster("dimer", h=0.6, fd_order=8)
    p = F.default_params(fd_order=8, precision=F.PREC_MIXED, tol_E=1e-7, tol_inner=1e-8)
    g = F.make_grid(*dims, 0.6, tuple(-0.3 * k for k in dims))
    E, _, st = ctx.solve(c.R, c.Z, c.h, p, grid=g)
    cv = _context(OFDFT_FD=0)
    Ev, _, sv = cv.solve(c.R, c.Z, c.h, p, grid=g)
    cv.close()
    assert st.converged and sv.converged
    assert abs(E - Ev) / c.M <= 1e-7


def test_mixed_corrections_hand_over_to_cg_at_the_rounding_floor(ctx):
    """A tolerance below what float-float residuals resolve: the direct corrections
    stop halving the residual, the CG form takes over, and the call ends with
    OFDFT_ENOTCONV and a potential at FP32 rounding, as the CG form alone does."""
    g = F.make_grid(36, 34, 33, 0.5)
    og = O.make_grid(36, 34, 33, 0.5, (0.0, 0.0, 0.0))
    phi_m = np.random.default_rng(2).standard_normal(g.shape)
    rho = (-O.laplacian(og, 6, phi_m) / (4.0 * np.pi)).astype(np.float32)
    sols = []
    cv = _context(OFDFT_FD=0)
    for c in (ctx, cv):
        c.reset_counters()
        phi = torch.zeros(g.shape, dtype=torch.float32, device=DEV)
        st = c.poisson(g, 12, phi, rho=torch.as_tensor(rho, device=DEV), tol=1e-18, max_it=40, allow_notconv=True)
        assert st.rel_residual > 1e-18 and st.iterations >= 3
        assert c.counters().kind_launches[F.K_CG_DIR_STENCIL] > 0
        sols.append(phi.double().cpu().numpy())
    cv.close()
    # both at their floors: equal to FP32 rounding (2^-24 each, doubled)
    assert np.linalg.norm(sols[0] - sols[1]) <= 2.0**-22 * np.linalg.norm(sols[1])


@pytest.mark.parametrize("ke,kh", [(-300, 0), (-80, 0), (80, 0), (300, 0), (0, -100), (0, 100), (-200, 60)])
def test_fp64_solves_do_not_depend_on_scale(ctx, ke, kh):
    """Sources and spacings scaled by powers of two far outside FP32's range: every
    operation of the solve scales exactly, so potential and steps are the unscaled
    ones bit for bit (phi ~ rho h^2)."""
    dims, order = (36, 40, 33), 12
    rho = np.random.default_rng(6).standard_normal(dims[::-1])

    def solve(ke, kh):
        g = F.make_grid(*dims, float(np.ldexp(0.6, kh)))
        phi = torch.zeros(g.shape, dtype=torch.float64, device=DEV)
        st = ctx.poisson(g, order, phi, rho=torch.as_tensor(np.ldexp(rho, ke), device=DEV), tol=1e-10, max_it=50)
        return np.ldexp(phi.cpu().numpy(), -ke - 2 * kh), st.iterations

    (p0, it0), (p1, it1) = solve(0, 0), solve(ke, kh)
    assert it0 == it1 and np.array_equal(p0, p1)


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), 1e30])
def test_mixed_solves_of_sources_that_are_not_finite_leave_the_potential(ctx, bad):
    """The corrections are launched before the host has seen the residual: a source
    that is not finite, or whose norm FP32 sums cannot hold, ends the call with
    OFDFT_ENONFINITE and the caller's potential as it was."""
    g = F.make_grid(36, 34, 33, 0.5)
    rho = torch.ones(g.shape, dtype=torch.float32, device=DEV)
    rho[3, 4, 5] = bad
    phi = torch.full(g.shape, 0.25, dtype=torch.float32, device=DEV)
    with pytest.raises(F.OfdftError, match="ENONFINITE"):
        ctx.poisson(g, 12, phi, rho=rho, tol=1e-8)
    assert bool((phi == 0.25).all())


@pytest.mark.parametrize("prec", [F.PREC_FP64, F.PREC_MIXED])
def test_evaluations_whose_poisson_solve_fails_write_no_gradient(ctx, prec):
    """The functional is launched behind the Poisson solve, before the host knows how it
    ended: where it fails (not converged, or not finite) grad and s stay as they were; and
    an evaluation at the potential as it is (solve_poisson=False) needs no convergence."""
    from paper_1405_6456_gb300 import workloads as W
    c = W.tiny_cluster("dimer", h=0.6, fd_order=8)
    dtype = torch.float64 if prec == F.PREC_FP64 else torch.float32
    g = F.make_grid(44, 36, 38, 0.6, (-13.2, -10.8, -11.4))
    b, u = (torch.empty(g.shape, dtype=dtype, device=DEV) for _ in range(2))
    Es = ctx.pseudocharge(g, 8, c.R, c.Z, b)
    ctx.initial_guess(g, c.R, c.Z, u)
    bad = u.clone()
    bad[5, 6, 7] = float("nan")

    def evaluate(uu, err=None, **kw):
        grad, s = torch.full_like(u, 7.0), torch.full_like(u, 7.0)
        solve = kw.pop("solve_poisson", True)
        p = F.default_params(fd_order=8, precision=prec, precond_rank1=0, **kw)
        args = (g, p, uu, b, torch.zeros_like(u), Es, 0.0, float("inf"), c.N, solve)
        if err is None:
            return ctx.energy_grad(*args, grad=grad, s=s), grad, s
        with pytest.raises(F.OfdftError, match=err):
            ctx.energy_grad(*args, grad=grad, s=s)
        assert bool((grad == 7.0).all()) and bool((s == 7.0).all())

    evaluate(u, "ENOTCONV", tol_poisson=1e-25, max_cg=1)
    evaluate(bad, "ENONFINITE", tol_poisson=1e-8)
    evaluate(bad, "ENONFINITE", tol_poisson=1e-8, solve_poisson=False)
    e, grad, s = evaluate(u, tol_poisson=1e-8, solve_poisson=False)
    # at phi = 0 the electrostatic term is absent from the gradient (and without a
    # penalty it does not depend on sum u^2, which other passes sum in other orders)
    e0, grad0, s0 = evaluate(u, terms=F.TERM_TF | F.TERM_VW | F.TERM_XC)
    assert e.poisson.rel_residual > 0.5 and torch.equal(grad, grad0) and torch.equal(s, s0)
