"""The atom kernels against the oracle where their tables and queues have edges:
nuclear widths and radii whose squared arguments cross the interval table's octaves
and leave it, boxes larger and smaller than the grid, atoms near and outside the
box's faces, every stencil radius."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
from paper_1405_6456_gb300 import build as B
from paper_1405_6456_gb300 import ofdft as F

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.build()
    c = F.Context(0)
    yield c
    c.close()


def _case(dims, h, seed):
    g = F.make_grid(*dims, h, tuple(-0.5 * n * h for n in dims))
    rng = np.random.default_rng(seed)
    half = 0.5 * h * np.array(dims)
    R = rng.uniform(-1.0, 1.0, (5, 3)) * half * 0.6
    R[1] = half - 0.1                      # at a corner
    R[2] = [half[0] + 1.0, 0.0, 0.2]       # outside the box
    R[3] = [-half[0] + 0.5 * h, 0.5 * h - half[1], 0.5 * h - half[2]]  # on a node
    return g, O.make_grid(*dims, h, tuple(g.origin)), R, np.array([3.0, 1.0, 2.0, 3.0, 0.5])


# (sigma, rc): the default; a wide nucleus inside one octave; a narrow one whose
# argument reaches 512 and leaves the table; a ball larger than the grid
@pytest.mark.parametrize("sigma,rc", [(1.0, 7.0), (2.5, 4.0), (0.25, 5.0), (0.9, 9.5)])
@pytest.mark.parametrize("dims,h,order", [((26, 21, 33), 0.6, 12), ((19, 24, 17), 0.8, 2), ((22, 30, 20), 0.7, 8)])
def test_pseudocharge_and_forces_match_oracle(ctx, sigma, rc, dims, h, order):
    g, og, R, Z = _case(dims, h, order)
    n = order // 2
    b = torch.empty(g.shape, dtype=torch.float64, device=DEV)
    es = ctx.pseudocharge(g, order, R, Z, b, sigma=sigma, rc=rc)
    b_ref, es_ref = O.pseudocharge(og, n, R, Z, sigma, rc)
    # b_J is a sum of 6n + 1 values of V / h^2 that cancel: rounding of V's scale
    scale = np.abs(O.lap_weights(n, h)).sum() * 6.0 * 3.0 * 2.0 / (sigma * np.sqrt(np.pi)) / (4.0 * np.pi)
    assert np.abs(b.cpu().numpy() - b_ref).max() <= 5 * 4e-16 * scale
    assert es == pytest.approx(es_ref, rel=1e-12)
    phi = 0.01 * np.random.default_rng(3).standard_normal(g.shape)
    for variant in (F.FORCE_PAPER, F.FORCE_EXACT):
        Fd = ctx.forces(g, order, R, Z, torch.as_tensor(phi, device=DEV), sigma=sigma, rc=rc, variant=variant)
        Fo = O.forces(og, n, R, Z, phi, sigma=sigma, rc=rc, exact=(variant == F.FORCE_EXACT))
        np.testing.assert_allclose(Fd, Fo, rtol=1e-10, atol=1e-11 * np.abs(Fo).max())


@pytest.mark.parametrize("gs,cut", [(2.0, 8.0), (0.7, 2.3), (5.0, 60.0)])
@pytest.mark.parametrize("dims,h", [((26, 21, 33), 0.6), ((64, 9, 8), 0.5)])
def test_initial_guess_matches_oracle(ctx, gs, cut, dims, h):
    g, og, R, Z = _case(dims, h, 7)
    u = torch.empty(g.shape, dtype=torch.float64, device=DEV)
    ctx.initial_guess(g, R, Z, u, guess_sigma=gs, guess_cut=cut)
    u_ref = O.initial_guess(og, R, Z, gs, cut)
    # three exponentials multiplied against one of the sum: a few units of 2^-53
    assert np.abs(u.cpu().numpy() - u_ref).max() <= 1e-14 * np.abs(u_ref).max()


@pytest.mark.parametrize("variant", [F.FORCE_PAPER, F.FORCE_EXACT])
def test_forces_of_balls_without_nodes_are_zero(ctx, variant):
    g, _, R, Z = _case((26, 21, 33), 0.6, 12)
    phi = torch.ones(g.shape, dtype=torch.float64, device=DEV)
    for rc in (0.0, -0.3, -1.0, -50.0):
        assert not ctx.forces(g, 12, R, Z, phi, rc=rc, variant=variant).any()


def test_forces_of_point_charges_and_negative_widths(ctx):
    """ofdft_forces takes any width: sigma = 0 is V = -Z/r (as any width far below the
    nearest node's distance), and erf is odd, so -sigma is the charge -Z."""
    dims, h = (26, 21, 33), 0.6
    g, og, R, Z = _case(dims, h, 12)
    R, Z = R[:2] + 0.07, Z[:2]
    phi = 0.01 * np.random.default_rng(3).standard_normal(g.shape)
    for sigma, ref in ((0.0, dict(sigma=1e-3)), (-0.25, dict(sigma=0.25))):
        Fd = ctx.forces(g, 12, R, Z, torch.as_tensor(phi, device=DEV), sigma=sigma, rc=5.0)
        Fo = O.forces(og, 6, R, -Z if sigma < 0 else Z, phi, rc=5.0, **ref)
        np.testing.assert_allclose(Fd, Fo, rtol=1e-10, atol=1e-11 * np.abs(Fo).max())


@pytest.mark.parametrize("k", [-60, 66])
def test_atom_kernels_do_not_depend_on_the_unit_of_length(ctx, k):
    """Lengths scaled by a power of two whose squares FP32 cannot hold: the FP32 screens
    only ever keep more, and the FP64 values scale exactly (b ~ 1/length^3, its self
    energy ~ 1/length; the forces' sums, in another order, to rounding)."""
    dims, h = (26, 21, 33), 0.6
    phi = np.random.default_rng(3).standard_normal(dims[::-1])

    def run(s):
        g, _, R, Z = _case(dims, h, 12)
        g = F.make_grid(*dims, h * s, tuple(x * s for x in g.origin))
        b = torch.empty(g.shape, dtype=torch.float64, device=DEV)
        es = ctx.pseudocharge(g, 12, R * s, Z, b, sigma=s, rc=7.0 * s)
        Fd = ctx.forces(g, 12, R * s, Z, torch.as_tensor(phi / s, device=DEV), sigma=s, rc=7.0 * s)
        u = torch.empty(g.shape, dtype=torch.float64, device=DEV)
        ctx.initial_guess(g, R * s, Z, u, guess_sigma=2.0 * s, guess_cut=8.0 * s)
        return b.cpu().numpy() * s**3, es * s, Fd * s**2, u.cpu().numpy() * s**1.5

    (b0, e0, f0, u0), (b1, e1, f1, u1) = run(1.0), run(2.0**k)
    assert np.array_equal(b0, b1) and e0 == pytest.approx(e1, rel=1e-14)
    np.testing.assert_allclose(f1, f0, rtol=1e-12, atol=1e-13 * np.abs(f0).max())
    # the guess's norm is a power, rounded apart at either scale: a few units of 2^-53
    np.testing.assert_allclose(u1, u0, rtol=1e-14, atol=0.0)
