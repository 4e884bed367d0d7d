"""Models whose neighbouring points differ by several line widths in velocity (a large
`dshift_frac` inserts no points between them): a point at the floor next to one at line centre.
Against the oracle, FP64 within 1e-10 and mixed precision within 1e-4."""
import numpy as np
import pytest

import synthetic as syn
from oracle import Oracle
from helpers import rel_err, gpu_context

pytestmark = pytest.mark.gpu


def _models():
    yield syn.model_clumpy_3d(n=120, seed=5, nside=1, n_lev=3, n_q=33)
    m = syn.model_clumpy_3d(n=120, seed=6, nside=1, n_q=20, species=syn.species_ladder(2))
    m.T = np.full(m.n, 3.0)
    yield m


@pytest.mark.parametrize("dshift_frac", [1.0, 3.0, 30.0])
@pytest.mark.parametrize("kind", ["step", "band1", "band2", "scatter", "image"])
def test_large_steps(kind, dshift_frac):
    band = int(kind[4:]) if kind.startswith("band") else 0
    tol = 1e-4 if kind == "mixed" else 1e-10
    for m in _models():
        o = Oracle(m, nthreads=16, dshift_frac=dshift_frac)
        p = o.lte()
        ctx = gpu_context(m, oracle_dirs=o.dirs, precision=int(kind == "mixed"), spectrum=1, alo_band=band,
                          dshift_frac=dshift_frac)
        ctx.trace_rays()
        ctx.set_populations(p)
        if kind == "image":
            u = np.linspace(-1e4, 1e4, 49)
            I, _ = ctx.image(4, 0, u)
            assert np.max(rel_err(I, o.image(p, 4, 0, u)[0])) < tol
            continue
        if kind == "scatter":
            xs = 3e-14 * m.n_coll / m.n_coll.max()
            ctx.set_scattering(xs, tol=1e-30, max_iter=2)
            Jo, Lo, Eo, Sp, _ = o.formal_solve_scattering(p, xs, tol=1e-30, max_iter=2)
        elif band:
            Jo, Lo, Eo, Mo = o.formal_solve_band(p, band)
            Eo = Eo[0]
        else:
            Jo, Lo, Eo, Sp = o.formal_solve(p, None, spectrum=True)
        ctx.formal_solve()
        J, L, E = ctx.get_radiation()
        assert np.max(rel_err(J, Jo)) < tol
        if band:
            # (terms below 1e-250 come from profiles that underflow in the oracle)
            assert np.max(rel_err(ctx.get_band_terms()[1], Mo, floor=1e-250)) < tol
        else:
            assert np.max(rel_err(ctx.get_spectrum(), Sp)) < tol
        if kind != "mixed":
            assert np.max(rel_err(L, Lo, floor=1e-300)) < tol and np.max(np.abs(E - Eo) / Jo) < tol


@pytest.mark.parametrize("dshift_frac", [2.0, 5.0, 30.0])
def test_large_steps_mixed(dshift_frac):
    for m in _models():
        o = Oracle(m, nthreads=16, dshift_frac=dshift_frac)
        Jo, Lo, Eo, Sp = o.formal_solve(o.lte(), None, spectrum=True)
        ctx = gpu_context(m, oracle_dirs=o.dirs, precision=1, spectrum=1, dshift_frac=dshift_frac)
        ctx.trace_rays()
        ctx.init_populations()
        ctx.formal_solve()
        assert np.max(rel_err(ctx.get_radiation()[0], Jo)) < 1e-4
        assert np.max(rel_err(ctx.get_spectrum(), Sp)) < 1e-4
