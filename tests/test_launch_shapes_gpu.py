"""The launch shapes and routes chosen by size, at the edges of their ranges: the FP32 formal
solve in every launch shape valid for a number of lines and bins, the statistical
equilibrium with a lane group per cell and a thread per cell, the network's row tiles,
and ray tracing into storage that is used again."""
import copy

import numpy as np
import pytest

import synthetic as syn
from oracle import Oracle
from oracle import mlp as omlp
from helpers import rel_err, gpu_context
from test_mlp_gpu import bf16

pytestmark = pytest.mark.gpu
TOL_MIX = 1e-4
N_SHAPES = 40


@pytest.mark.parametrize("L,Q", [(1, 7), (1, 33), (2, 8), (2, 16), (3, 17), (3, 9), (4, 24), (5, 25), (4, 32), (5, 33),
                                 (6, 48), (3, 49), (7, 64), (2, 65), (1, 128)])
def test_every_valid_shape(L, Q):
    """Lanes without a bin, lines beyond the last group, and one to four bins per lane and
    line: radiation field and mean intensity per bin within the mixed tolerance."""
    m = syn.model_clumpy_3d(n=120, seed=Q, n_lev=L + 1, n_q=Q, nside=1)
    o = Oracle(m, nthreads=16)
    p0 = o.lte()
    Jo, Lo, Eo, Sp = o.formal_solve(p0, None, spectrum=True)
    ctx = gpu_context(m, oracle_dirs=o.dirs, precision=1, spectrum=1)
    ctx.trace_rays()
    ctx.set_populations(p0)
    for v in range(-1, N_SHAPES):   # a shape that does not fit L x Q runs as the default one
        ctx.set_variant(v)
        ctx.formal_solve()
        J, Lam, E = ctx.get_radiation()
        assert np.max(rel_err(J, Jo)) < TOL_MIX, v
        assert np.max(np.abs(E - Eo) / Jo) < TOL_MIX, v
        assert np.max(np.abs(Lam - Lo)) < TOL_MIX * max(1e-6, float(np.max(Lo))), v
        assert np.max(rel_err(ctx.get_spectrum(), Sp)) < TOL_MIX, v
    best, ms, tried = ctx.autotune(reps=1)
    assert tried >= 1 and np.max(rel_err(ctx.get_radiation()[0], Jo)) < TOL_MIX


# 1e-10 as for the other tests of this update; the oracle's pivoted LU adds an error of some
# hundred roundings of the largest population to the others
@pytest.mark.parametrize("n_lev,n", [(2, 3999), (2, 4000), (3, 31), (5, 33), (8, 129), (9, 65), (12, 100), (13, 40),
                                     (20, 70), (24, 37), (25, 21), (33, 20), (40, 23)])
@pytest.mark.parametrize("twice", [False, True])
def test_statistical_equilibrium_routes(n_lev, n, twice):
    """Cells that do not fill a block, the numbers of cells on both sides of the line between
    the two kernels, and (twice) a second line on a pair of levels, whose rates add up."""
    m = syn.model_clumpy_3d(n=n, seed=n_lev, n_lev=n_lev, nside=1, n_q=5)
    if twice:
        sp = m.species = copy.copy(m.species)
        sp.up, sp.lo = np.append(sp.up, sp.up[0]), np.append(sp.lo, sp.lo[0])
        sp.A = np.append(sp.A, 0.5 * sp.A[0])
    o = Oracle(m, nthreads=8)
    ctx = gpu_context(m, oracle_dirs=o.dirs)
    ctx.init_populations()
    rng = np.random.default_rng(n)
    shape = (m.n, m.species.n_lines)
    J = 1e-16 * 10.0 ** rng.uniform(-3, 2, shape)
    L = rng.uniform(0, 0.999, shape)
    E = J * rng.uniform(0.01, 1, shape)
    ctx.set_radiation(J, L, E)
    ctx.update_populations()
    ref, nf = o.stateq(J, L, E)
    assert ctx.status_counts()[0] == nf
    assert np.all(np.abs(ctx.get_populations() - ref) <= 1e-10 * ref.clip(0) + 1e-13 * m.n_spec[:, None])


def _gradient(theta, X, Y, n_out):
    """The oracle's backpropagation through the GPU's forward roundings (BF16 activations and
    weights of the 128-wide layers), so that the same units are active."""
    W1, b1, W2, b2, W3, b3, W4, b4 = omlp.unpack(theta.astype(np.float64), n_out)
    W2, W3, W4 = (bf16(w).astype(np.float64) for w in (W2, W3, W4))
    h1 = bf16(np.maximum(X @ W1 + b1, 0)).astype(np.float64)
    h2 = bf16(np.maximum(h1 @ W2 + b2, 0)).astype(np.float64)
    h3 = bf16(np.maximum(h2 @ W3 + b3, 0)).astype(np.float64)
    z = h3 @ W4 + b4
    z = z - z.max(1, keepdims=True)
    logp = z - np.log(np.exp(z).sum(1, keepdims=True))
    mask = Y >= omlp.FRAC_MIN
    d = np.where(mask, logp - np.log(np.maximum(Y, omlp.FRAC_MIN)), 0.0)
    g = 2.0 * d / max(int(mask.sum()), 1)
    dz = g - np.exp(logp) * g.sum(1, keepdims=True)
    d3 = (dz @ W4.T) * (h3 > 0)
    d2 = (d3 @ W3.T) * (h2 > 0)
    d1 = (d2 @ W2.T) * (h1 > 0)
    return [X.T @ d1, d1.sum(0), h1.T @ d2, d2.sum(0), h2.T @ d3, d3.sum(0), h3.T @ dz, dz.sum(0)]


@pytest.mark.parametrize("rows", [1, 63, 64, 65, 300])
@pytest.mark.parametrize("n_out", [2, 16, 17, 32])
def test_network_gradient_at_tile_edges(rows, n_out):
    """Each of up to three BF16 roundings of a gradient on its way back is 2^-9 at most, so
    three are below 1e-2 of each block's norm; 2e-2 leaves room for the activations'
    roundings at the last bit."""
    import paper_1912_08445_gb300 as mg
    rng = np.random.default_rng(100 * rows + n_out)
    theta = omlp.init_params(n_out, 9).astype(np.float32)
    X = rng.normal(size=(rows, 4)).astype(np.float32)
    Y = rng.dirichlet(np.ones(n_out), size=rows).astype(np.float32)
    net = mg.MLP(n_out, seed=3)
    net.set_params(theta)
    net.set_normalisation(np.zeros(4, np.float32), np.ones(4, np.float32))
    for rep in range(2):   # the second call finds the workspace of the first
        loss, g = net.loss_grad(X, Y)
        k = 0
        for b in _gradient(theta, X.astype(np.float64), Y.astype(np.float64), n_out):
            a = g[k:k + b.size].astype(np.float64)
            k += b.size
            assert np.linalg.norm(a - b.ravel()) <= 2e-2 * np.linalg.norm(b), (rep, b.shape)


def test_tracing_again_into_kept_storage():
    """Tracing twice, on another stream, and tracing a longer and a shorter set of rays one
    after the other gives the rays of a fresh context, element by element."""
    import torch
    small, big = syn.model_clumpy_3d(n=200, seed=1, nside=1), syn.model_clumpy_3d(n=900, seed=2, nside=2)
    def rays(ctx, m):
        R = 12 * m.nside ** 2
        return [ctx.get_ray(o, r) for o in range(0, m.n, 37) for r in range(R)]
    want = {}
    for k, m in (("small", small), ("big", big)):
        c = gpu_context(m)
        c.trace_rays()
        want[k] = rays(c, m)
    ctx = gpu_context(small)
    ctx.trace_rays()
    side = torch.cuda.Stream()
    for k, m in (("big", big), ("small", small), ("small", small), ("big", big)):
        ctx.load_model(m)
        if k == "small":
            ctx.set_stream(side.cuda_stream)
        ctx.trace_rays()
        for a, b in zip(rays(ctx, m), want[k]):
            assert all(np.array_equal(a[f], b[f]) for f in ("cells", "nsub", "ds", "vpar"))
    ctx.set_stream(None)
    ctx.trace_rays()
    for a, b in zip(rays(ctx, big), want["big"]):
        assert all(np.array_equal(a[f], b[f]) for f in ("cells", "nsub", "ds", "vpar"))
