"""Every form the persistent solver kernels take as the SMs they may use shrink, against the oracle's steps.

The forms follow from the rows an SM gets, so max_sms walks through them on one small hierarchy: the hybridized CG with
four, two or one lane a row and its entries in shared memory, with two rows a lane streamed from memory, and with its
state in memory. A Krylov iterate after k steps is fixed by the method (oracle.krylov), so every form must give it; the
bound is the one the step-parity tests of the same kernels use (FP64 recurrences over 14 steps).
"""
import numpy as np
import pytest

from oracle import coarse, hierarchy, krylov
from synth.grids import problem_config

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
