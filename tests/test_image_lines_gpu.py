"""The image kernels for up to four lines in reach at the edges of their splits, against the
oracle (1e-10 in FP64 contexts, 1e-4 in mixed ones): channel counts around the warp and the
block, one to five lines in reach (five take the general kernel), pairs longer than one
staging, a density jump of ten decades between neighbours, a floor too large for lists."""
import numpy as np
import pytest

import synthetic as syn
from oracle import Oracle
from helpers import rel_err, gpu_context

pytestmark = pytest.mark.gpu
TOL = {0: 1e-10, 1: 1e-4}


def _check(m, precision, u, rays=(0, 5), origins=None, line=0, **opts):
    o = Oracle(m, nthreads=16, **{k: v for k, v in opts.items() if k == "chi_min"})
    ctx = gpu_context(m, oracle_dirs=o.dirs, precision=precision, **opts)
    ctx.trace_rays()
    ctx.init_populations()
    sel = slice(None) if origins is None else origins
    for r in rays:
        I, xy = ctx.image(r, line, u)
        Io, xyo = o.image(o.lte(), r, line, u, origins=origins)
        assert np.max(rel_err(I[sel], Io)) < TOL[precision], r


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n_ch", [1, 2, 31, 33, 64, 65, 257])
def test_channel_counts(n_ch, precision):
    _check(syn.model_clumpy_3d(n=150, seed=3, nside=1, n_lev=3), precision, np.linspace(-9e3, 8e3, n_ch))


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n_lev", [2, 3, 4, 5, 6])
def test_lines_in_reach(n_lev, precision):
    m = syn.model_clumpy_3d(n=150, seed=12, nside=1, species=syn.species_ladder(n_lev))
    _check(m, precision, np.linspace(-3e3, 3e3, 40), line=n_lev - 2)


@pytest.mark.parametrize("precision", [0, 1])
def test_pairs_longer_than_a_staging(precision):
    # 30 widths per cell: pairs of ~900 points
    m = syn.vz_problem1(abundance=1e-6, v_inf=5e4, n_shells=50)
    _check(m, precision, np.linspace(-6e4, 6e4, 61), origins=np.arange(0, 50, 7))


def test_density_jump():
    # (FP64 contexts: the FP32 image's weight at an element's own cell is rounded)
    m = syn.model_clumpy_3d(n=200, seed=8, nside=1, n_lev=3)
    dense = np.random.default_rng(1).random(m.n) < 0.2
    m.n_spec = np.where(dense, m.n_spec, 1e-10 * m.n_spec)
    m.T = np.where(dense, 10.0, 160.0)
    _check(m, 0, np.linspace(-1.2e4, 1.2e4, 64))


@pytest.mark.parametrize("precision", [0, 1])
def test_large_floor(precision):
    _check(syn.model_clumpy_3d(n=150, seed=4, nside=1, n_lev=3), precision, np.linspace(-5e3, 5e3, 33), chi_min=1e-18)
