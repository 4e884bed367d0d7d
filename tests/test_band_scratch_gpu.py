"""The band ALO's coupling terms where their scratch (at most 1 GiB) covers a part of the origins
at a time, and where there is no room for it: within 1e-10 of the oracle either way."""
import numpy as np
import pytest

import synthetic as syn
from oracle import Oracle
from helpers import FullDevice, rel_err, gpu_context

pytestmark = pytest.mark.gpu
TOL = 1e-10


@pytest.fixture(scope="module")
def model():
    # 2 chunks of bins x 4 lines x 3072 rays x 2 terms x 8 bytes an origin: 2730 origins in 1 GiB
    m = syn.model_clumpy_3d(n=2800, seed=6, n_lev=5, n_q=2, nside=16)
    origins = np.array([0, 1, 1365, 2728, 2729, 2730, 2731, 2799])
    o = Oracle(m, nthreads=16)
    return m, o, origins, o.formal_solve_band(o.lte(), 2, origins=origins)


def _context(m, o):
    ctx = gpu_context(m, oracle_dirs=o.dirs, precision=0, alo_band=2)
    ctx.trace_rays()
    ctx.init_populations()
    return ctx


def _compare(ctx, origins, want):
    Jo, Lo, Eo, Mo = want
    J, L, E = ctx.get_radiation()
    Jb, M = ctx.get_band_terms()
    assert np.max(rel_err(J[origins], Jo)) < TOL and np.max(rel_err(L[origins], Lo, floor=1e-300)) < TOL
    for got, ref in ((E, Eo[0]), (Jb[0], Eo[1]), (Jb[1], Eo[2]), (M, Mo)):
        assert np.max(rel_err(got[origins], ref, floor=1e-300)) < TOL


def test_origins_in_parts(model):
    m, o, origins, want = model
    ctx = _context(m, o)
    ctx.formal_solve()
    _compare(ctx, origins, want)


def test_no_room_for_the_scratch(model):
    """With the memory for the coupling terms themselves and half of the scratch left, the
    solve still succeeds."""
    m, o, origins, want = model
    ctx = _context(m, o)
    terms = m.n * 3072 * 2 * (8 * 4 + 16)      # coupling terms and geometry of the band points
    with FullDevice(terms + (1 << 29)):
        ctx.formal_solve()
        _compare(ctx, origins, want)
