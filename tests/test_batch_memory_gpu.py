"""A batch without memory for its Ng history reports MG_ERR_OOM, and iterates once there is some."""
import numpy as np
import pytest

import synthetic as syn
from helpers import FullDevice
import paper_1912_08445_gb300 as mg
from paper_1912_08445_gb300.binding import MG_ERR_OOM

pytestmark = pytest.mark.gpu


def test_no_room_for_the_history():
    # 400k points without neighbours, 20 levels: 64 MB an iterate. The first update from any
    # populations is the solution (no light but the boundary's), so a batch that starts from it
    # stops at once and needs no history.
    n, n_lev = 400_000, 20
    rng = np.random.default_rng(0)
    sp = syn.species_rotor(n_lev, rng)
    models = []
    for _ in range(2):
        ctx = mg.Context(precision=1)
        ctx.set_mesh(rng.normal(size=(n, 3)), np.zeros((n, 3)), np.zeros(n + 1, np.int64), np.zeros(0, np.int32),
                     np.ones(n, np.uint8))
        ctx.set_species(sp.E, sp.g, sp.mass, sp.up, sp.lo, sp.A, sp.T_grid, sp.K_down)
        ctx.set_model(np.full(n, 1e9), np.full(n, 50.0), np.full(n, 100.0), np.full(n, 1e3))
        ctx.set_directions(1)
        ctx.set_quadrature(5)
        ctx.trace_rays()
        ctx.init_populations()
        ctx.formal_solve()
        ctx.update_populations()
        models.append(ctx)
    batch = mg.Batch(models)
    reps, _ = batch.iterate()
    assert all(r["iterations"] == 1 for r in reps)
    for ctx in models:
        ctx.init_populations()
    with FullDevice(32 << 20):
        with pytest.raises(mg.MagritteError) as e:
            batch.iterate()
        assert e.value.code == MG_ERR_OOM
    for ctx in models:
        ctx.init_populations()
    reps, _ = batch.iterate()
    assert all(r["converged"] for r in reps)
