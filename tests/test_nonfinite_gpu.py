"""Populations that are not finite stay visible in FP64 results: not finite on the rays that meet
such a cell, the same bits as before elsewhere."""
import numpy as np
import pytest

import synthetic as syn
from helpers import rel_err, gpu_context

pytestmark = pytest.mark.gpu


def _seen(ctx, m, cell, rays):
    """Origins with `cell` on one of the rays, or next to one (interpolated points)."""
    hit = np.zeros(m.n, bool)
    for o in range(m.n):
        for r in rays:
            hit[o] |= o == cell or cell in ctx.get_ray(o, r)["cells"]
    return hit


@pytest.mark.parametrize("value", [np.nan, np.inf])
@pytest.mark.parametrize("scatter", [False, True])
def test_formal_solve(value, scatter):
    """One cell's populations replaced: J and J_eff of every line are not finite at the origins
    whose rays meet the cell, and as before at the others."""
    m = syn.model_clumpy_3d(n=300, seed=3, n_lev=3, nside=1)
    ctx = gpu_context(m, precision=0)
    ctx.trace_rays()
    ctx.init_populations()
    def solve():
        if scatter:
            ctx.set_scattering(3e-14 * m.n_coll / m.n_coll.max(), tol=1e-30, max_iter=1)
        ctx.formal_solve()
        return ctx.get_radiation()

    J0, L0, E0 = solve()
    cell = int(np.argmax(m.is_bdy == 0))
    p = ctx.get_populations()
    p[cell] = value
    ctx.set_populations(p)
    J, L, E = solve()
    hit = _seen(ctx, m, cell, range(12))
    assert hit.any() and not hit.all()
    assert not np.isfinite(J[hit]).any() and not np.isfinite(E[hit]).any()
    assert np.array_equal(J[~hit], J0[~hit]) and np.array_equal(E[~hit], E0[~hit])


@pytest.mark.parametrize("value", [np.nan, np.inf])
@pytest.mark.parametrize("n_lev", [2, 4])
def test_image(value, n_lev):
    """One and three lines in reach: in the channels that the cell's line profile reaches, the
    rays through the cell are not finite, other rays are as before."""
    m = syn.model_clumpy_3d(n=300, seed=3, nside=1, v_max=0.0, species=syn.species_ladder(n_lev))
    ctx = gpu_context(m, precision=0)
    ctx.trace_rays()
    ctx.init_populations()
    u = np.linspace(-400.0, 400.0, 33)
    I0, _ = ctx.image(5, 0, u)
    p = ctx.get_populations()
    cell = int(np.argmax(m.is_bdy == 0))
    p[cell] = value
    ctx.set_populations(p)
    I, _ = ctx.image(5, 0, u)
    anti = ctx.get_directions()[1]
    hit = _seen(ctx, m, cell, [5, int(anti[5])])
    assert hit.any() and not hit.all()
    assert not np.isfinite(I[hit]).any()
    assert np.max(rel_err(I[~hit], I0[~hit])) == 0.0
