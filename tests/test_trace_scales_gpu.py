"""Ray tracing of models with many scales, whose FP32 bounds must hold and stay tight near the
centre: rays bit for bit the oracle's, and a time that follows the number of cells crossed."""
import numpy as np
import pytest

import synthetic as syn
from oracle import Oracle
from helpers import compare_rays, gpu_context

pytestmark = pytest.mark.gpu


def _cloud(n, decades, nside, centre=0.0):
    """A cloud with radii spread evenly over `decades` of the radius, around a point `centre`
    outer radii from the origin of the coordinates."""
    m = syn.model_clumpy_3d(n=n, seed=7, nside=nside)
    rng = np.random.default_rng(7)
    inner = m.is_bdy == 0
    k = int(inner.sum())
    d = rng.normal(size=(k, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    m.pos[inner] = 0.98e15 * (10.0 ** rng.uniform(-decades, 0.0, k))[:, None] * d
    m.nbr_off, m.nbr_idx = syn.knn_symmetric(m.pos, 16)
    m.vel = 1e3 * m.pos / np.linalg.norm(m.pos, axis=1)[:, None]
    m.pos = m.pos + centre * 1e15
    return m


@pytest.mark.parametrize("decades,centre", [(2, 0.0), (5, 0.0), (9, 0.0), (3, 30.0)])
def test_rays_match_oracle(decades, centre):
    m = _cloud(1500, decades, 1, centre)
    o = Oracle(m, nthreads=16)
    ctx = gpu_context(m, oracle_dirs=o.dirs)
    ctx.trace_rays()
    origins = np.arange(0, m.n, 3)
    assert compare_rays(ctx, o.trace_all(origins), origins, 12) == []


def test_time_follows_the_cells():
    """Five decades of radius cost at most three times a cloud of one decade, per cell crossed
    (decisions in FP64 near the centre cost 7.5 times)."""
    t = []
    for decades in (1, 5):
        ctx = gpu_context(_cloud(20000, decades, 2), precision=1, profile=1)
        ctx.trace_rays()
        ctx.reset_kernel_times()
        for _ in range(3):
            st, _ = ctx.trace_rays()
        ms, launches = ctx.kernel_times()["trace_count"]
        t.append(ms / launches / st["n_elements"])
    assert t[1] < 3.0 * t[0]
