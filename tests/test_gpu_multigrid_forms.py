"""The multigrid preconditioner's kernels over the mode counts and level sizes that choose between them.

A cell's block takes one to eight modes (a group of lanes a block, padded where a level's mode counts differ), the
levels of at most 512 unknowns are one precomputed map, and the coarsest level's inverse is formed by a cluster
whatever its order. The cases put the map's boundary on both sides of level 1 (63 cells of 8 modes are 504 unknowns,
213 cells of 3 are 639), leave it nothing but the coarsest level (63 cells of one mode end the cycle at level 1), have
odd and mixed mode counts, and aggregates of level-1 cells both small (residual and restriction in one kernel) and
large (two kernels). One application is compared with the oracle's FP64 cycle: FP32 rounding (6e-8) times the
conditioning of the cell blocks (at most 5.3e3 here) or of the coarsest matrix (at most 2.2e4) is at most 1.3e-3, and
2e-3 is taken; a wrong index or a lost term shows at 1e-1. The Picard update must meet its own tolerance on the
oracle's matrix, in the oracle's number of steps to a tenth.
"""
import numpy as np
import pytest

from oracle import hierarchy, newton, precond, tpfa
from synth.grids import problem_config

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,scale,agg,modes", [("chan3d_64", 16, [64, 8, 8], [1, 1, 1]),
                                                  ("chan3d_64", 16, [64, 8, 8], [8, 8, 8]),
                                                  ("chan3d_64", 24, [64, 8, 8], [1, 1, 1]),
                                                  ("chan3d_64", 24, [64, 8, 8], [3, 3, 3]),
                                                  ("chan3d_64", 24, [64, 8, 8], [6, 5, 2]),
                                                  ("chan3d_64", 21, [48, 6, 6], [7, 4, 4]),
                                                  ("chan3d_64", 24, [8, 27, 8], [2, 2, 2]),
                                                  ("cart2d_32", 32, [16, 4, 4], [2, 3, 2])])
def test_mode_counts_and_level_sizes(nlmg_lib, name, scale, agg, modes):
    pr = problem_config(name, scale=scale)
    pr.opts = dict(pr.opts, lin_precond=1, n_levels=3, agg_size=agg, modes=modes)
    ctx = nlmg_lib.Context(pr.mesh, pr.kappa_kind, pr.kappa_a, pr.opts)
    ctx.set_data(pr.f_cell, pr.g_face)
    rng = np.random.default_rng(71)
    p = rng.uniform(0, 1, pr.mesh.n_cells)
    A = newton.picard_matrix(pr.mesh, pr.kappa_kind, pr.kappa_a, p).tocsr()
    H = hierarchy.build(pr.mesh, precond.extended_options(pr.opts))
    lv = precond.build(A, H, precond.levels_for(H))
    r = rng.uniform(-1, 1, pr.mesh.n_cells)
    ref = precond.vcycle(lv, H, r)
    assert np.linalg.norm(ctx.precond_apply(p, r) - ref) <= 2e-3 * np.linalg.norm(ref)

    R = tpfa.reduced_residual(pr.mesh, pr.kappa_kind, pr.kappa_a, p, pr.f_cell, pr.g_face)
    S = 1.0 / np.sqrt(A.diagonal())
    ctx.set_options(lin_tol=1e-8, lin_maxit=500)
    dx, it = ctx.picard_update(0, p)
    _, it_ref = precond.pcg(A, -R, lambda q: precond.vcycle(lv, H, q), 500, tol=1e-8, w=S)
    assert np.linalg.norm(S * (A @ dx + R)) <= 1e-8 * (1 + 1e-6) * np.linalg.norm(S * R)
    assert abs(it - it_ref) <= 1 + it_ref // 10
