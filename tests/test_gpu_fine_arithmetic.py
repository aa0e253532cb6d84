"""Rounding and range of the level-0 operators: transmissibilities, the exact Jacobian and the Newton system's solver."""
import numpy as np
import pytest

from oracle import tpfa
from synth.grids import cartesian_mesh

pytestmark = pytest.mark.gpu


def context(nlmg_lib, mesh, kind, a, g=None, f=None, **opts):
    ctx = nlmg_lib.Context(mesh, kind, a, dict(dict(n_levels=1), **opts))
    ctx.set_data(np.zeros(mesh.n_cells) if f is None else f, np.zeros(mesh.n_faces) if g is None else g)
    return ctx


def checkerboard(shape):
    return (np.indices(shape).sum(0) % 2).T.reshape(-1).astype(float)


@pytest.mark.parametrize("k0", [3.0, 0.3, 0.7, 2.7, 9.9, 11.0, 19.4, 49.0, 7e5, 1e-3])
def test_transmissibilities_of_a_uniform_field_are_exact(nlmg_lib, k0):
    """Where both halves of a face are the same number u and kappa = 1, the transmissibility u / 2 is a number of the
    format, and with pressures 0 and 1 in turn so is every flux. A cell adds up to four of them, whole multiples of u / 2,
    with at most three roundings."""
    mesh = cartesian_mesh((9, 9), np.full(81, k0))
    u = k0 / 3.0
    mesh.half_trans[:] = np.where(mesh.half_trans > 0, u, 0.0)
    ctx = context(nlmg_lib, mesh, 0, 0.0)
    p = checkerboard((9, 9))
    K, L = mesh.face_cells[tpfa.flux_dofs(mesh)].T
    flux = np.where(L >= 0, u / 2 * (p[K] - p[L]), u * p[K])
    np.testing.assert_array_equal(ctx.fine_flux(p), flux)
    want = np.zeros(81)
    np.add.at(want, K, np.where(L >= 0, p[K] - p[L], 2 * p[K]))
    np.add.at(want, L[L >= 0], -(p[K] - p[L])[L >= 0])
    np.testing.assert_allclose(ctx.fine_residual(p), want * (u / 2), rtol=3 * 2.0 ** -53, atol=0)


def divided_residual(mesh, kind, a, p, g):
    """The residual by the transmissibility ha (hb / (ha + hb)) of the two kappa-scaled halves, f = 0."""
    with np.errstate(all="ignore"):
        k = tpfa.kappa(p, kind, a)
        K, L = mesh.face_cells.T
        ha, hb = k[K] * mesh.half_trans[:, 0], k[L] * mesh.half_trans[:, 1]
        T = np.where(mesh.face_bc == 0, ha * (hb / (ha + hb)), np.where(mesh.face_bc == 1, ha, 0.0))
        flux = np.where(mesh.face_bc == 2, 0.0, T * (p[K] - np.where(mesh.face_bc == 0, p[L], g)))
        r = np.zeros(mesh.n_cells)
        np.add.at(r, K, flux)
        np.add.at(r, L[mesh.face_bc == 0], -flux[mesh.face_bc == 0])
    return r, flux[mesh.face_bc != 2]


@pytest.mark.parametrize("shift", [-760.0, -720.0, -709.9, -500.0, -300.0, 300.0, 500.0, 700.0, 720.0])
@pytest.mark.parametrize("cells", ["all", "one", "dirichlet"])
def test_residual_keeps_its_range(nlmg_lib, shift, cells):
    """kappa = exp(p) from zero to overflow, in all cells or in one: the residual and the fluxes are what the kappa-scaled
    halves give, to the rounding of a subnormal kappa (2^-35 of it at -720), and infinities and NaN stand where they give
    them."""
    if cells == "dirichlet":
        mesh = cartesian_mesh((1, 1), np.array([1.7]))
        base = np.array([0.25])
    else:
        rng = np.random.default_rng(9)
        mesh = cartesian_mesh((5, 4), rng.uniform(0.5, 2.0, 20))
        base = rng.integers(-200, 200, 20) / 1024.0
    where = np.zeros(mesh.n_cells, bool)
    where[slice(None) if cells == "all" else 7 % mesh.n_cells] = True
    p = base + np.where(where, shift, 0.0)
    g = np.where(mesh.face_bc == 1, 0.5 if cells != "all" else shift + 0.5, 0.0)
    want, flux = divided_residual(mesh, 0, 1.0, p, g)
    ctx = context(nlmg_lib, mesh, 0, 1.0, g)
    scale = np.abs(np.where(np.isfinite(want), want, 0.0)).max()
    np.testing.assert_allclose(ctx.fine_residual(p), want, rtol=1e-9, atol=1e-9 * scale)
    np.testing.assert_allclose(ctx.fine_flux(p), flux, rtol=1e-9, atol=1e-9 * scale)


@pytest.mark.parametrize("shift", [-600, -500, -400, 400, 500, 600])
def test_newton_update_does_not_depend_on_the_size_of_kappa(nlmg_lib, shift):
    """kappa = exp(p): a shift of p and g scales the residual and the Jacobian by the same number, so the update is the
    same (pressures are multiples of 1/1024, so the shift is exact; the linear solves stop at 1e-12 of the residual and
    the scaled matrix has a condition below 1e3)."""
    rng = np.random.default_rng(4)
    mesh = cartesian_mesh((6, 5), rng.uniform(0.5, 2.0, 30))
    p = rng.integers(0, 1024, 30) / 1024.0
    g = rng.integers(0, 1024, mesh.n_faces) / 1024.0
    dx = []
    for s in (0, shift):
        ctx = context(nlmg_lib, mesh, 0, 1.0, np.where(mesh.face_bc == 1, g + s, 0.0), newton_lin_tol=1e-12, lin_maxit=200)
        dx.append(ctx.newton_update(p + s)[0])
    assert np.linalg.norm(dx[1] - dx[0]) <= 1e-9 * np.linalg.norm(dx[0])


@pytest.mark.parametrize("power", [150, 260, 300])
def test_newton_update_scales_with_large_pressures(nlmg_lib, power):
    """kappa = 1 / (1 + p^2) is p^-2 to the last bit from 2^30 on, where scaling p by a power of two scales the update by
    it."""
    rng = np.random.default_rng(6)
    mesh = cartesian_mesh((6, 5), rng.uniform(0.5, 2.0, 30))
    p = rng.uniform(1.0, 1.5, 30) * 2.0 ** 30
    g = np.where(mesh.face_bc == 1, rng.uniform(1.0, 1.5, mesh.n_faces) * 2.0 ** 30, 0.0)
    dx = []
    for s in (1.0, 2.0 ** (power - 30)):
        ctx = context(nlmg_lib, mesh, 1, 0.0, s * g, newton_lin_tol=1e-12, lin_maxit=200)
        dx.append(ctx.newton_update(s * p)[0] / s)
    assert np.linalg.norm(dx[1] - dx[0]) <= 1e-9 * np.linalg.norm(dx[0])


def test_bicgstab_stops_at_its_tolerance_where_a_step_gains_much(nlmg_lib):
    """Nearly decoupled cells: the first step leaves about 2^-16 of (s, s). The stopping test has to see (r, r) to a part
    in 1e12 (rounding of the residual's entries, 2^-53 of s, gives about 5e-14), so a tolerance just above or below the
    residual after one step decides whether there is a second."""
    for seed in range(12):
        rng = np.random.default_rng(seed)
        mesh = cartesian_mesh((2, 40), np.ones(80))
        inner = mesh.face_bc == 0
        mesh.half_trans[inner] *= 1e-5 * rng.uniform(0.5, 1.5, (inner.sum(), 1))
        p = rng.uniform(0, 1, 80)
        g = np.zeros(mesh.n_faces)
        J = tpfa.reduced_jacobian(mesh, 0, 0.0, p, g).toarray()
        R = tpfa.reduced_residual(mesh, 0, 0.0, p, np.zeros(80), g)
        S = 1.0 / np.sqrt(np.maximum(np.diag(J), 0.5 * tpfa.picard_diagonal(mesh, 0, 0.0, p)).astype(np.longdouble))
        A, r = J * S[:, None] * S[None, :], -S * R
        v = A @ r
        alpha = (r @ r) / (r @ v)
        s = r - alpha * v
        t = A @ s
        r1 = s - (t @ s) / (t @ t) * t
        assert (r1 @ r1) < 2.0 ** -15 * (s @ s)
        tol = float(np.sqrt((r1 @ r1) / (r @ r)))
        for factor, steps in ((1 + 5e-13, {1}), (1 - 5e-13, {2, 3})):
            ctx = context(nlmg_lib, mesh, 0, 0.0, g, newton_lin_tol=tol * factor, lin_maxit=50)
            assert ctx.newton_update(p)[1] in steps, (seed, factor)
