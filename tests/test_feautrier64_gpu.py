"""The FP64 formal solve of lines that do not overlap (warp-autonomous kernel) at the edges
of its splits, against the oracle within 1e-10: bins that leave lanes idle, straddle warps
or need several chunks per line; one to sixteen warps per origin; few and many ray pairs;
the band terms of a line spread over chunks; rescaling of very thick columns; inverted
populations (the opacity floor keeps the line's emission); a floor too large for far
points to be left out; density jumps of ten decades between neighbours."""
import numpy as np
import pytest

import synthetic as syn
from oracle import Oracle
from helpers import rel_err, gpu_context

pytestmark = pytest.mark.gpu
TOL = 1e-10


def _check(m, pops=None, band=0, **opts):
    o = Oracle(m, nthreads=16, **{k: v for k, v in opts.items() if k == "chi_min"})
    ctx = gpu_context(m, oracle_dirs=o.dirs, precision=0, spectrum=1, alo_band=band, **opts)
    ctx.trace_rays()
    p0 = o.lte() if pops is None else pops(o.lte())
    ctx.set_populations(p0)
    ctx.formal_solve()
    J, L, E = ctx.get_radiation()
    if band:
        Jo, Lo, Eo, Mo = o.formal_solve_band(p0, band)
        Jb, M = ctx.get_band_terms()
        for b in range(band):
            assert np.max(rel_err(Jb[b], Eo[b + 1], floor=1e-300)) < TOL
        assert np.max(rel_err(M, Mo, floor=1e-300)) < TOL
        Eo = Eo[0]
    else:
        Jo, Lo, Eo, Jn = o.formal_solve(p0, None, spectrum=True)
        assert np.max(rel_err(ctx.get_spectrum(), Jn)) < TOL
    assert np.max(rel_err(J, Jo)) < TOL and np.max(rel_err(E, Eo)) < TOL
    assert np.max(rel_err(L, Lo, floor=1e-300)) < TOL


@pytest.mark.parametrize("n_lev,n_q,nside", [(2, 1, 1), (2, 31, 2), (2, 32, 1), (2, 33, 1), (3, 16, 1), (4, 11, 2),
                                            (4, 40, 1), (6, 63, 1), (9, 70, 1), (20, 5, 1), (3, 100, 1)])
def test_bins_and_lines(n_lev, n_q, nside):
    _check(syn.model_clumpy_3d(n=150, seed=n_q, n_lev=n_lev, n_q=n_q, nside=nside))


@pytest.mark.parametrize("n", [60, 900])
def test_few_and_many_origins(n):
    _check(syn.model_clumpy_3d(n=n, seed=9, n_lev=3, n_q=21, nside=1))


@pytest.mark.parametrize("band", [1, 2])
@pytest.mark.parametrize("n_lev,n_q", [(3, 40), (4, 70), (5, 9)])
def test_band_terms_over_chunks(n_lev, n_q, band):
    _check(syn.model_clumpy_3d(n=120, seed=5, n_lev=n_lev, n_q=n_q, nside=1), band=band)


def test_thick_columns_are_rescaled():
    m = syn.model_sphere_1d(n=120, seed=2)
    m.n_spec = m.n_spec * 3e6
    _check(m)


def test_inverted_populations():
    def invert(p):
        q = p.copy()
        q[:, 1] = 40.0 * q[:, 0]
        return q
    _check(syn.model_clumpy_3d(n=150, seed=3, n_lev=3, nside=1), invert)


def test_large_floor():
    _check(syn.model_clumpy_3d(n=150, seed=4, n_lev=3, nside=1), chi_min=1e-18)


def test_density_and_temperature_jumps():
    m = syn.model_clumpy_3d(n=200, seed=8, nside=1, n_lev=3)
    dense = np.random.default_rng(1).random(m.n) < 0.2
    m.n_spec = np.where(dense, m.n_spec, 1e-10 * m.n_spec)
    m.T = np.where(dense, 10.0, 160.0)
    _check(m)
