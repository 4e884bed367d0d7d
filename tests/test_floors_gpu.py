"""The floors of the transfer and a dark boundary, against the oracle: an optical-depth floor
`dtau_min` that counts in every interval, and a boundary intensity that underflows to zero,
against which any emission counts. FP64 within 1e-10 (the step, both band widths, scattering,
images), mixed precision within 1e-4."""
import numpy as np
import pytest

import synthetic as syn
from oracle import Oracle
from helpers import rel_err, gpu_context

pytestmark = pytest.mark.gpu
TOL = {0: 1e-10, 1: 1e-4}
KINDS = ["step", "band1", "band2", "scatter", "image"]


def _cloud():
    return syn.model_clumpy_3d(n=150, seed=3, n_lev=3, nside=1)


def _invert(p):
    q = p.copy()
    q[:, 1] = 40.0 * q[:, 0]
    return q


def _check(m, kind, pops=None, precision=0, scattering=3e-14, **opts):
    """One result of the kind, from LTE populations or pops(LTE populations)."""
    tol = TOL[precision]
    band = int(kind[4:]) if kind.startswith("band") else 0
    o = Oracle(m, nthreads=16, **{k: v for k, v in opts.items() if k in ("chi_min", "dtau_min", "T_cmb")})
    p0 = o.lte() if pops is None else pops(o.lte())
    ctx = gpu_context(m, oracle_dirs=o.dirs, precision=precision, spectrum=1, alo_band=band, **opts)
    ctx.trace_rays()
    ctx.set_populations(p0)
    if kind == "image":
        u = np.linspace(-1.1e4, 1.1e4, 65)
        for line in range(m.species.n_lines):
            I, _ = ctx.image(5, line, u)
            assert np.isfinite(I).all()
            Io, _ = o.image(p0, 5, line, u)
            # (the oracle's emissivity times profile is a subnormal number, good to 2^-1075, where
            # the intensity it gives over up to 1e15 m is below 1e-298)
            assert np.max(rel_err(I, Io, floor=1e-298)) < tol
        return
    if kind == "scatter":
        xs = scattering * m.n_coll / m.n_coll.max()
        ctx.set_scattering(xs, tol=1e-30, max_iter=3)
        Jo, Lo, Eo, Sp, _ = o.formal_solve_scattering(p0, xs, tol=1e-30, max_iter=3)
    elif band:
        Jo, Lo, Eo, Mo = o.formal_solve_band(p0, band)
    else:
        Jo, Lo, Eo, Sp = o.formal_solve(p0, None, spectrum=True)
    ctx.formal_solve()
    J, L, E = ctx.get_radiation()
    assert np.isfinite(J).all() and np.isfinite(L).all() and np.isfinite(E).all()
    if band:
        Jb, M = ctx.get_band_terms()
        for b in range(band):
            assert np.max(rel_err(Jb[b], Eo[b + 1], floor=1e-300)) < tol
        assert np.max(rel_err(M, Mo, floor=1e-300)) < tol
        Eo = Eo[0]
    else:
        assert np.max(rel_err(ctx.get_spectrum(), Sp)) < tol
    assert np.max(rel_err(J, Jo)) < tol
    if precision == 0:
        assert np.max(rel_err(E, Eo, floor=1e-300)) < tol and np.max(rel_err(L, Lo, floor=1e-300)) < tol


@pytest.mark.parametrize("dtau_min", [1e-12, 1e-9, 1e-6])
@pytest.mark.parametrize("kind", KINDS)
def test_optical_depth_floor(kind, dtau_min):
    """Every interval has at least the optical depth dtau_min, those of far points too."""
    _check(_cloud(), kind, dtau_min=dtau_min)


def test_optical_depth_floor_of_promoted_cells():
    """Cells solved again in FP64 in a mixed-precision context: all of them here."""
    _check(_cloud(), "step", precision=1, dtau_min=1e-3, tau_fp64=1.000001)


# Planck's function is exactly zero at 5 mK for these lines (near 100 GHz) and a normal number
# at 50 mK
@pytest.mark.parametrize("T_cmb", [5e-3, 5e-2])
@pytest.mark.parametrize("inverted", [False, True])
@pytest.mark.parametrize("kind", KINDS)
def test_dark_boundary(kind, inverted, T_cmb):
    """Against a boundary without light any emission counts, that of inverted lines (whose
    opacity is at the floor) too. (Inverted lines without scattering: their opacity would
    cancel against it.)"""
    _check(_cloud(), kind, _invert if inverted else None, T_cmb=T_cmb, scattering=0.0 if inverted else 3e-14)


@pytest.mark.parametrize("dtau_min", [1e-4, 1e-2])
@pytest.mark.parametrize("variant", [13, 15])   # one line, and two, per warp; every point swept
def test_optical_depth_floor_of_every_interval_mixed(variant, dtau_min):
    m = _cloud()
    o = Oracle(m, nthreads=16, dtau_min=dtau_min)
    Jo, Lo, Eo, Sp = o.formal_solve(o.lte(), None, spectrum=True)
    ctx = gpu_context(m, oracle_dirs=o.dirs, precision=1, spectrum=1, dtau_min=dtau_min)
    ctx.trace_rays()
    ctx.init_populations()
    ctx.set_variant(variant)
    ctx.formal_solve()
    assert np.max(rel_err(ctx.get_radiation()[0], Jo)) < TOL[1]
    assert np.max(rel_err(ctx.get_spectrum(), Sp)) < TOL[1]


@pytest.mark.parametrize("dtau_min", [1e-4, 1e-2])
def test_optical_depth_floor_mixed(dtau_min):
    """The default launch shape, then every shape with and without far-wing skipping."""
    m = _cloud()
    _check(m, "step", precision=1, dtau_min=dtau_min)
    o = Oracle(m, nthreads=16, dtau_min=dtau_min)
    Jo = o.formal_solve(o.lte())[0]
    ctx = gpu_context(m, oracle_dirs=o.dirs, precision=1, dtau_min=dtau_min)
    ctx.trace_rays()
    ctx.init_populations()
    for v in range(40):
        ctx.set_variant(v)
        ctx.formal_solve()
        assert np.max(rel_err(ctx.get_radiation()[0], Jo)) < TOL[1], v


@pytest.mark.parametrize("chi_min", [1e-36, 1e-40, 1e-60])
def test_tiny_opacity_floor_of_an_fp32_image(chi_min):
    """Floors that are not normal FP32 numbers."""
    _check(_cloud(), "image", precision=1, chi_min=chi_min)


@pytest.mark.parametrize("chi_min", [1e-36, 1e-40, 1e-48])
def test_tiny_opacity_floor_of_inverted_lines_in_an_fp32_image(chi_min):
    """An inverted line has its emissivity over the floor as its source function."""
    _check(_cloud(), "image", _invert, precision=1, chi_min=chi_min)


def _no_emission(p):
    """Upper levels empty in two cells of three: those only absorb."""
    q = p.copy()
    q[np.random.default_rng(1).random(p.shape[0]) < 0.67, 1:] = 0.0
    return q


@pytest.mark.parametrize("overlap", [False, True])
@pytest.mark.parametrize("kind", KINDS)
def test_bright_background_behind_cold_cells(kind, overlap):
    """Intensities far below the boundary's, to which points at the floor still add."""
    m = _cloud()
    if overlap:
        m.species = syn.species_ladder(4)
    m.n_spec = 1e3 * m.n_spec
    _check(m, kind, _no_emission, T_cmb=1500.0)
