"""Which form of the level-0 Krylov kernels ran, as the SMs they may use shrink.

The profile's algorithmic bytes of a launch count the vectors its form moves (registers: two an iteration, the FP64 CG in
memory 12, the FP32 one 11; BiCGStab 4 and 19), so they tell the form. The expected one follows from the slices of 32
cells a warp gets: blocks of up to 15 warps, at least four slices a block, and a power of two of blocks up to 8.
"""
import numpy as np
import pytest

from synth.grids import problem_config, voronoi_problem

pytestmark = pytest.mark.gpu


def slices_a_warp(nslice, sms):
    grid = min(sms, (nslice + 3) // 4)
    if nslice <= 64:
        grid = min(grid, 8)
    if grid <= 8:
        up = 1 << (grid - 1).bit_length()
        grid = up if up <= sms else grid
    per = -(-nslice // grid)
    return -(-per // min(15, per))


@pytest.mark.parametrize("scale", [12, 24])
def test_registers_wherever_the_cells_fit(nlmg_lib, scale):
    pr = problem_config("chan3d_64", scale=scale)
    ctx = nlmg_lib.Context(pr.mesh, pr.kappa_kind, pr.kappa_a, dict(pr.opts, n_levels=1))
    ctx.set_data(pr.f_cell, pr.g_face)
    n, nnz = pr.mesh.n_cells, 2 * int((pr.mesh.face_bc == 0).sum())
    p = np.random.default_rng(3).uniform(0, 1, n)
    seen = set()
    for sms in (1, 2, 3, 4, 6, 8, 15, 29, 152):
        R = slices_a_warp((n + 31) // 32, sms)
        for precision, most, in_memory in ((0, 5, 12), (1, 9, 11)):
            ctx.set_options(lin_precision=precision, lin_tol=1e-6, lin_maxit=6, max_sms=sms)
            ctx.profile(True)
            _, it = ctx.picard_update(0, p)
            _, _, moved, _ = ctx.profile_read(0)
            ctx.profile(False)
            v, registers = (4, 8)[precision == 0], R <= most
            per_it = (4 + v) * nnz + (2 if registers else in_memory) * v * n
            extra = 1 if registers or precision == 0 else 0   # the pipelined forms' product at the start
            assert moved == (16 + 3 * v + 16) * n + (it + extra) * per_it, (sms, R, precision)
            seen.add((precision, registers))
        ctx.set_options(lin_precision=0, newton_lin_tol=1e-12, lin_maxit=5, max_sms=sms)
        ctx.profile(True)
        _, it = ctx.newton_update(p)
        _, _, moved, _ = ctx.profile_read(3)
        ctx.profile(False)
        assert moved == 80 * n + it * (24 * nnz + 16 * n + (4 if R <= 4 else 19) * 8 * n), (sms, R)
        seen.add((2, R <= 4))
    assert len(seen) == (6 if scale == 24 else 3)


def test_fp64_rows_beyond_shared_memory_run_in_memory(nlmg_lib):
    """On a Voronoi mesh (rows of some 25 entries) on two SMs a warp has five slices or fewer, but the rows do not fit
    beside each other in shared memory: the FP64 CG runs in memory then, the FP32 CG and the BiCGStab stream the rows."""
    pr = voronoi_problem(14)
    ctx = nlmg_lib.Context(pr.mesh, pr.kappa_kind, pr.kappa_a, dict(pr.opts, n_levels=1))
    ctx.set_data(pr.f_cell, pr.g_face)
    inner = pr.mesh.face_bc == 0
    n, nnz = pr.mesh.n_cells, 2 * int(inner.sum())
    widest = int(np.bincount(pr.mesh.face_cells[inner].reshape(-1)).max())
    p = np.random.default_rng(3).uniform(0.4, 0.6, n)
    forms = {}
    for sms in (2, 0):
        R = slices_a_warp((n + 31) // 32, sms or 152)
        grid = min(sms or 152, ((n + 31) // 32 + 3) // 4)
        warps = min(15, -(-((n + 31) // 32) // grid))
        fits = warps * R * 32 * (12 * widest + 8) <= 218 * 1024
        for precision, v, in_memory in ((0, 8, 12), (1, 4, 11)):
            ctx.set_options(lin_precision=precision, lin_tol=1e-6, lin_maxit=6, max_sms=sms)
            ctx.profile(True)
            _, it = ctx.picard_update(0, p)
            _, _, moved, _ = ctx.profile_read(0)
            ctx.profile(False)
            registers = R <= (5, 9)[precision] and (fits or precision == 1)
            per_it = (4 + v) * nnz + (2 if registers else in_memory) * v * n
            assert moved == (16 + 3 * v + 16) * n + (it + 1) * per_it, (sms, R, precision)
            forms[sms, precision] = registers
    assert forms == {(2, 0): False, (2, 1): True, (0, 0): True, (0, 1): True}
