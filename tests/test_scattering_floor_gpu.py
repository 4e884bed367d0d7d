"""Scattering beside points whose line opacity is at the floor (FP64), against the oracle within
1e-10."""
import numpy as np
import pytest

import synthetic as syn
from oracle import Oracle
from helpers import rel_err, gpu_context

pytestmark = pytest.mark.gpu
TOL = 1e-10


@pytest.mark.parametrize("model", ["sphere", "cloud"])
def test_patchy_scattering(model):
    """Cells that scatter beside cells that do not: the source function of a point at the floor
    enters with the opacity of the scattering point after it, in every bin."""
    if model == "sphere":
        m = syn.model_sphere_1d(n=30, seed=4, n_q=63)
    else:
        m = syn.model_clumpy_3d(n=100, seed=4, n_q=16, nside=1, n_lev=6)
    m.T = 30.0 * m.T
    xs = 1e-16 * (np.random.default_rng(3).random(m.n) < 0.7)
    o = Oracle(m, nthreads=16)
    p0 = o.lte()
    for T_cmb in (2.725, 50.0):
        o = Oracle(m, nthreads=16, T_cmb=T_cmb)
        ctx = gpu_context(m, oracle_dirs=o.dirs, precision=0, spectrum=1, T_cmb=T_cmb)
        ctx.trace_rays()
        ctx.set_populations(p0)
        ctx.set_scattering(xs, tol=1e-30, max_iter=2)
        ctx.formal_solve()
        J, L, E = ctx.get_radiation()
        Jo, Lo, Eo, Sp, _ = o.formal_solve_scattering(p0, xs, tol=1e-30, max_iter=2)
        assert np.max(rel_err(J, Jo)) < TOL and np.max(rel_err(E, Eo)) < TOL
        assert np.max(rel_err(L, Lo, floor=1e-300)) < TOL
        assert np.max(rel_err(ctx.get_spectrum(), Sp)) < TOL
