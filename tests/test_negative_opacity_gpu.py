"""Negative line opacities (inverted populations) where they add to other opacity before the
floor: FP64, against the oracle within 1e-10."""
import numpy as np
import pytest

import synthetic as syn
from oracle import Oracle
from helpers import rel_err, gpu_context

pytestmark = pytest.mark.gpu
TOL = 1e-10


@pytest.mark.parametrize("n_lev", [3, 4, 5])
@pytest.mark.parametrize("level", [1, 2])
def test_image_of_overlapping_lines(n_lev, level):
    """One line of two to four in reach is inverted (weakly and strongly): its opacity takes
    from that of the others."""
    m = syn.model_clumpy_3d(n=150, seed=12, nside=1, species=syn.species_ladder(n_lev))
    o = Oracle(m, nthreads=16)
    u = np.linspace(-3e3, 3e3, 40)
    for factor in (1.05, 3.0):
        p = o.lte()
        p[:, level] = factor * p[:, level - 1] * (2 * level + 1.0) / (2 * level - 1.0)
        ctx = gpu_context(m, oracle_dirs=o.dirs, precision=0)
        ctx.trace_rays()
        ctx.set_populations(p)
        for ray in (0, 5):
            I, _ = ctx.image(ray, 0, u)
            Io, _ = o.image(p, ray, 0, u)
            assert np.max(rel_err(I, Io)) < TOL


def test_scattering_with_an_inverted_line():
    """An inverted line's opacity takes from the scattering opacity, by up to a twentieth (so
    that no sum is ill-conditioned)."""
    m = syn.model_clumpy_3d(n=150, seed=3, n_lev=3, nside=1)
    o = Oracle(m, nthreads=16)
    p = o.lte()
    p[:, 1] = 3.0 * p[:, 0] * m.species.g[1] / m.species.g[0]
    h, c = 6.62607015e-34, 299792458.0
    sp = m.species
    nu = (sp.E[1] - sp.E[0]) / h
    Bul = sp.A[0] * c ** 2 / (2 * h * nu ** 3)
    chi = h * nu / (4 * np.pi) * (p[:, 0] * sp.g[1] / sp.g[0] - p[:, 1]) * Bul
    peak = chi * c / (nu * np.sqrt(np.pi) * np.array([o.width(k) for k in range(m.n)]))
    xs = np.full(m.n, 20.0 * np.abs(peak).max())
    ctx = gpu_context(m, oracle_dirs=o.dirs, precision=0, spectrum=1)
    ctx.trace_rays()
    ctx.set_populations(p)
    ctx.set_scattering(xs, tol=1e-30, max_iter=3)
    ctx.formal_solve()
    J, L, E = ctx.get_radiation()
    Jo, Lo, Eo, Sp, _ = o.formal_solve_scattering(p, xs, tol=1e-30, max_iter=3)
    assert np.max(rel_err(J, Jo)) < TOL and np.max(rel_err(ctx.get_spectrum(), Sp)) < TOL
    assert np.max(np.abs(E - Eo) / Jo) < TOL and np.max(np.abs(L - Lo)) < TOL
