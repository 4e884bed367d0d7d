"""The ray store of a context over a loop of models: up to 1 GiB is kept while the model changes
and used again by the next trace, with the rays of a fresh context element by element; more
is given back at once, and what is kept where memory runs short."""
import numpy as np
import pytest

import synthetic as syn
from helpers import FullDevice, gpu_context
import paper_1912_08445_gb300 as mg

pytestmark = pytest.mark.gpu


def _free():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def _rays(ctx, m):
    return [ctx.get_ray(o, r) for o in range(0, m.n, 97) for r in range(0, 12 * m.nside ** 2, 5)]


def _same(a, b):
    return all(np.array_equal(x[f], y[f]) for x, y in zip(a, b) for f in ("cells", "nsub", "ds", "vpar"))


def test_kept_over_models():
    """About 100 MB of rays: smaller and larger models within the store's room, one beyond it,
    and one that leaves it mostly empty."""
    ctx = gpu_context(syn.model_clumpy_3d(n=3000, seed=1, nside=2))
    ctx.trace_rays()
    for n in (2500, 2990, 3400, 900, 2000):
        m = syn.model_clumpy_3d(n=n, seed=n, nside=2)
        before = _free()
        ctx.load_model(m)
        assert abs(_free() - before) < 30 << 20, n      # the store is still there
        with pytest.raises(mg.MagritteError):
            ctx.get_ray(0, 0)                           # and holds no rays of this model
        ctx.trace_rays()
        fresh = gpu_context(m)
        fresh.trace_rays()
        assert _same(_rays(ctx, m), _rays(fresh, m)), n


def test_large_store_is_given_back():
    big = syn.model_clumpy_3d(n=12000, seed=2, nside=4)
    ctx = gpu_context(big)
    st, _ = ctx.trace_rays()
    assert 32 * st["n_elements"] > 1 << 30
    before = _free()
    ctx.load_model(syn.model_clumpy_3d(n=500, seed=3, nside=1))
    assert _free() - before > 31 * st["n_elements"]


def test_kept_store_gives_way():
    """With less memory left than a second model's fields need, they take the kept store's."""
    m = syn.model_clumpy_3d(n=3000, seed=1, nside=2)
    # 600k points without neighbours: 14 MB each of positions and velocities, 24 MB of other fields
    n = 600_000
    pos = np.random.default_rng(0).normal(size=(n, 3))
    zero = np.zeros(n)
    ctx = gpu_context(m)
    ctx.trace_rays()
    with FullDevice(32 << 20):
        ctx.set_mesh(pos, np.zeros((n, 3)), np.zeros(n + 1, np.int64), np.zeros(0, np.int32), np.ones(n, np.uint8))
        ctx.set_model(zero + 1e10, zero + 20.0, zero + 100.0, zero + 1e4)
