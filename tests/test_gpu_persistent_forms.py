"""Every form the persistent solver kernels take as the SMs they may use shrink, against the oracle's steps.

The forms follow from the rows an SM gets, so max_sms walks through them on one small hierarchy: the hybridized CG with
four, two or one lane a row and its entries in shared memory, with two rows a lane streamed from memory, and with its
state in memory; the level-0 CG (FP64, FP32) and BiCGStab with one to as many slices a warp as they take, in memory, and
on a mesh of wide rows (a Voronoi tessellation) whose rows do not fit in shared memory. A Krylov iterate after k steps is
fixed by the method (oracle.krylov), so every form must give it; the bounds are those the step-parity tests of the same
kernels use (FP64 recurrences over 14 steps 1e-9, FP32 over 7 steps 2e-4, BiCGStab over 6 steps 1e-9).
"""
import numpy as np
import pytest

from oracle import coarse, fas, hierarchy, krylov, newton, tpfa
from synth.grids import problem_config, voronoi_problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def setup(nlmg_lib):
    pr = problem_config("chan3d_64", scale=24)
    opts = dict(pr.opts, n_levels=3, agg_size=[64, 8, 8], modes=[4, 4, 4])
    H = hierarchy.build(pr.mesh, opts)
    ctx = nlmg_lib.Context(pr.mesh, pr.kappa_kind, pr.kappa_a, opts)
    ctx.set_data(pr.f_cell, pr.g_face)
    return pr, H, ctx


@pytest.mark.parametrize("max_sms", [1, 2, 4, 24, 48, 0])
@pytest.mark.parametrize("tight", [False, True], ids=["pipelined", "two_synchronisations"])
def test_coarse_step_forms_follow_the_oracle(setup, max_sms, tight):
    pr, H, ctx = setup
    k, tol = 14, 1e-9 if tight else 1e-6
    ctx.set_options(coarse_lin_tol=tol, coarsest_lin_tol=tol, lin_maxit=k, max_sms=max_sms)
    for l in (1, 2):
        lev = H.levels[l]
        rng = np.random.default_rng(60 + l)
        x = rng.uniform(-0.5, 0.5, lev.n_flux + lev.n_p)
        b = rng.uniform(-1, 1, lev.n_flux + lev.n_p)
        nf = lev.n_flux
        dx, it = ctx.picard_update(l, x, b)
        r = coarse.operator(lev, pr.kappa_kind, pr.kappa_a, x[:nf], x[nf:]) - b
        ref, it_ref = krylov.hybridized(lev, pr.kappa_kind, pr.kappa_a, x[:nf], x[nf:], -r, k=k)
        assert it == it_ref == k
        assert np.linalg.norm(dx - ref) <= 1e-9 * np.linalg.norm(ref)


@pytest.fixture(scope="module", params=["cartesian", "voronoi"])
def fine(request, nlmg_lib):
    if request.param == "cartesian":
        pr = problem_config("chan3d_64", scale=24)
        opts = dict(pr.opts, n_levels=3, agg_size=[64, 8, 8], modes=[4, 4, 4])
        sms = [1, 4, 6, 8, 10, 15, 29, 0]   # 13,824 cells: in memory, then 5, 4, 3, 2 slices a warp and one
    else:
        pr = voronoi_problem(8)
        opts = dict(pr.opts)
        sms = [1, 2, 0]
    ctx = nlmg_lib.Context(pr.mesh, pr.kappa_kind, pr.kappa_a, opts)
    ctx.set_data(pr.f_cell, pr.g_face)
    # between the data's solution at half the nonlinearity and itself (see the step-parity tests)
    p = newton.solve(pr.mesh, pr.kappa_kind, 0.5 * pr.kappa_a, pr.f_cell, pr.g_face)[0]
    p = p + 0.05 * np.random.default_rng(31).uniform(-1, 1, pr.mesh.n_cells)
    R = tpfa.reduced_residual(pr.mesh, pr.kappa_kind, pr.kappa_a, p, pr.f_cell, pr.g_face)
    return pr, ctx, opts, p, R, sms


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "fp32"])
def test_fine_cg_forms_follow_the_oracle(fine, precision):
    pr, ctx, opts, p, R, sms = fine
    A = newton.picard_matrix(pr.mesh, pr.kappa_kind, pr.kappa_a, p)
    k, tol = (14, 1e-9) if precision == 0 else (7, 2e-4)
    ref, _ = krylov.jacobi_pcg(A, -R, k)
    for m in sms:
        ctx.set_options(lin_precision=precision, lin_tol=1e-6, lin_maxit=k, max_sms=m)
        dx, it = ctx.picard_update(0, p)
        assert it == k, m
        assert np.linalg.norm(dx - ref) <= tol * np.linalg.norm(ref), m


def test_fine_bicgstab_forms_follow_the_oracle(fine):
    pr, ctx, opts, p, R, sms = fine
    J = tpfa.reduced_jacobian(pr.mesh, pr.kappa_kind, pr.kappa_a, p, pr.g_face)
    S = fas.FAS(hierarchy.build(pr.mesh, opts), pr.mesh, pr.kappa_kind, pr.kappa_a, pr.f_cell, pr.g_face, opts)
    ref, _ = krylov.bicgstab_scaled(J, -R, 1.0 / S.jacobi_diag(p), 6)
    for m in sms:
        ctx.set_options(lin_precision=0, newton_lin_tol=1e-12, lin_maxit=6, max_sms=m)
        dx, it = ctx.newton_update(p)
        assert it == 6, m
        assert np.linalg.norm(dx - ref) <= 1e-9 * np.linalg.norm(ref), m


@pytest.mark.parametrize("cells", [1, 3])
def test_fine_bicgstab_meets_its_tolerance_where_the_residual_collapses(nlmg_lib, cells):
    """A system of very few unknowns is solved to rounding within as many steps, so (r, r) falls far below (s, s) in one
    step and is summed from the vectors: the tolerance is still met."""
    from synth.grids import cartesian_mesh
    mesh = cartesian_mesh((cells, 1), np.array([1.0, 20.0, 0.3])[:cells])
    g = np.where(mesh.face_bc == 1, np.where(np.arange(mesh.n_faces) % 2 == 0, 1.0, 0.2), 0.0)
    ctx = nlmg_lib.Context(mesh, 0, 1.0, dict(n_levels=1, newton_lin_tol=1e-13, lin_maxit=50))
    ctx.set_data(np.zeros(cells), g)
    p = np.linspace(0.9, 0.3, cells)
    dx, it = ctx.newton_update(p)
    J = tpfa.reduced_jacobian(mesh, 0, 1.0, p, g)
    R = tpfa.reduced_residual(mesh, 0, 1.0, p, np.zeros(cells), g)
    assert 1 <= it <= 2 * cells + 2
    assert np.linalg.norm(J @ dx + R) <= 1e-12 * np.linalg.norm(R)
