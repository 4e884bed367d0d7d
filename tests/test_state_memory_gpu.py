"""A context without memory for its populations and line data reports MG_ERR_OOM, and solves once
there is some."""
import numpy as np
import pytest

import synthetic as syn
from helpers import FullDevice
import paper_1912_08445_gb300 as mg
from paper_1912_08445_gb300.binding import MG_ERR_OOM

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
def test_no_room_for_the_state(precision):
    # 500k points without neighbours, 20 levels: 80 MB of populations, twice, then 152 MB of
    # line data: the third allocation fails
    n, rng = 500_000, np.random.default_rng(0)
    sp = syn.species_rotor(20, rng)
    ctx = mg.Context(precision=precision)
    ctx.set_mesh(rng.normal(size=(n, 3)), np.zeros((n, 3)), np.zeros(n + 1, np.int64), np.zeros(0, np.int32),
                 np.ones(n, np.uint8))
    ctx.set_species(sp.E, sp.g, sp.mass, sp.up, sp.lo, sp.A, sp.T_grid, sp.K_down)
    ctx.set_model(np.full(n, 1e9), np.full(n, 50.0), np.full(n, 100.0), np.full(n, 1e3))
    ctx.set_directions(1)
    ctx.set_quadrature(5)
    ctx.trace_rays()
    with FullDevice(224 << 20):
        for _ in range(2):
            with pytest.raises(mg.MagritteError) as e:
                ctx.init_populations()
            assert e.value.code == MG_ERR_OOM
    ctx.init_populations()
    ctx.formal_solve()
    J, L, E = ctx.get_radiation()
    assert np.isfinite(J).all() and np.all(L == 0.0)
