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
