"""Workloads of this package for performance measurement: the calls a program makes on a
prepared model, over the range of models the package is used on.

  listed()             the fixed cases
  draw(rng)            one more case of the same ranges
  prepare(case, seed)  the context (or batch, or network) and device buffers a program holds
  run(state)           one pass through the public entry points
  exact(case, seed)    the same outputs in plain 64-bit torch
  work(case)           bytes and flops the pass cannot do without

Kinds of case:
  step      one ALI iteration from given populations: formal solve, then the population
            update; J, L, J_eff and the new populations come back
  ali       the whole accelerated Lambda iteration from LTE to convergence
  batch     the same for many small clouds in one batch
  snapshot  a freshly set mesh: ray tracing, LTE populations, first formal solve
  image     one image of a solved model along a ray direction
  grad      one loss and gradient evaluation of the network that proposes populations

Results of mixed-precision contexts are single-precision numbers and are returned as such.
"""
import math

import numpy as np
import torch

import paper_1912_08445_gb300 as mg
import synthetic as syn

H, KB, C = 6.62607015e-34, 1.380649e-23, 299792458.0
T_CMB, CHI_MIN, DTAU_MIN, DSHIFT = 2.725, 1e-30, 1e-30, 1.0 / 3.0


def _case(name, kind, model, n, nside, n_q, n_lev, fp64, **kw):
    return dict(name=name, kind=kind, model=model, n=n, nside=nside, n_q=n_q, n_lev=n_lev, fp64=fp64, **kw)


def listed():
    return [
        # the smallest model: the 1D spherical cloud (200 shells, 12 rays, 31 bins), where
        # latency and launches count; double precision
        _case("sphere_200", "step", "sphere", 200, 1, 31, 2, True),
        # double-precision step of a 3D cloud (5-level rotor, 4 lines x 31 bins, 48 rays)
        _case("cloud_fp64", "step", "cloud", 1500, 2, 31, 5, True),
        # the same with the tri-diagonal approximate Lambda operator (GMRES)
        _case("cloud_fp64_band", "step", "cloud", 600, 2, 31, 5, True, band=1),
        # scattering: the formal solve iterates on the mean intensity per bin
        _case("cloud_fp64_scatter", "step", "cloud", 200, 1, 31, 3, True, scatter=True),
        # mixed precision, the clumpy cloud at its full size, launch shape autotuned
        _case("cloud_mixed", "step", "cloud", 50000, 2, 31, 5, False, tuned=True),
        # mixed precision, the Keplerian disc: 192 rays, 20-level rotor, 19 lines x 63 bins
        _case("disc_mixed", "step", "disc", 32000, 4, 63, 20, False),
        # ALI to convergence of a model of the learned-start corpus (3000 points, 20 levels)
        _case("disc_small_ali", "ali", "disc", 3000, 2, 31, 20, False),
        # a parameter study: uneven clouds, solved together
        _case("batch_ali", "batch", "cloud", 1700, 1, 31, 5, False, models=8),
        # a new snapshot of a simulation: every call starts from an untraced mesh
        _case("snapshot", "snapshot", "cloud", 20000, 2, 31, 5, False),
        # images: 63 velocity channels of the disc in single precision, and of a cloud in
        # double precision
        _case("image_mixed", "image", "disc", 20000, 2, 63, 20, False),
        _case("image_fp64", "image", "cloud", 10000, 2, 41, 5, True),
        # one training batch of the network
        _case("network_grad", "grad", "rows", 4096, 0, 0, 20, False),
    ]


def _cost(c):
    """Relative cost of a case, for keeping drawn ones below the largest listed one."""
    u = c["n"] ** (4.0 / 3.0) * 12 * c["nside"] ** 2 * (c["n_lev"] - 1) * c["n_q"]
    return u * (250.0 if c["fp64"] else 1.0)


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    what = rng.choice(["sphere", "cloud64", "cloud64", "cloud", "cloud", "disc", "disc", "ali", "batch", "snapshot",
                       "image", "grad"])
    if what == "grad":
        return dict(kind="grad", model="rows", n=size(100, 8192), nside=0, n_q=0, n_lev=rng.randint(2, 32), fp64=False)
    if what == "sphere":
        return dict(kind="step", model="sphere", n=size(40, 300), nside=rng.choice([1, 2]), n_q=rng.randint(11, 100),
                    n_lev=2, fp64=True)
    n_q = rng.choice([31, 63, rng.randint(7, 64)])
    if what == "cloud64":
        c = dict(kind="step", model="cloud", n=size(100, 1500), nside=rng.choice([1, 2]), n_q=rng.randint(7, 40),
                 n_lev=rng.randint(2, 6), fp64=True)
        option = rng.choice(["", "band", "scatter"])
        if option == "band":
            c.update(band=rng.choice([1, 2]), n=min(c["n"], 600))
        if option == "scatter":
            c.update(scatter=True, nside=1, n=min(c["n"], 200))
        return c
    if what == "batch":
        return dict(kind="batch", model="cloud", n=size(300, 1700), nside=1, n_q=n_q, n_lev=rng.randint(2, 6),
                    fp64=False, models=rng.randint(2, 8))
    if what == "ali":
        return dict(kind="ali", model="disc", n=size(500, 3000), nside=rng.choice([1, 2]), n_q=31,
                    n_lev=rng.randint(5, 20), fp64=False)
    if what == "image":
        fp64 = rng.random() < 0.5
        return dict(kind="image", model=rng.choice(["cloud", "disc"]), n=size(500, 10000 if fp64 else 20000), nside=2,
                    n_q=rng.randint(5, 128), n_lev=rng.randint(3, 12), fp64=fp64)
    model = "disc" if what == "disc" else "cloud"
    c = dict(kind="snapshot" if what == "snapshot" else "step", model=model,
             n=size(1000, 20000 if what == "snapshot" else 32000 if model == "disc" else 50000),
             nside=rng.choice([1, 2, 4]) if model == "disc" else rng.choice([1, 2]), n_q=n_q,
             n_lev=rng.randint(5, 20) if model == "disc" else rng.randint(2, 8), fp64=False)
    most = _cost(listed()[5 if model == "disc" else 4])
    while _cost(c) > most:
        c["n"] = int(0.8 * c["n"])
    return c


# ------------------------------------------------------------------------- inputs
def _model(c, seed, n=None):
    n = c["n"] if n is None else n
    if c["model"] == "sphere":
        return syn.model_sphere_1d(n=n, seed=seed, n_q=c["n_q"], nside=c["nside"])
    if c["model"] == "disc":
        # the densities of the optically thick disc, and those of the corpus for the ALI
        dens, x = (1e12, 1e-5) if c["kind"] == "ali" else (2.5e16, 1e-4)
        return syn.model_disc(n=n, seed=seed, nside=c["nside"], n_q=c["n_q"], n_lev=c["n_lev"], n_h2_in=dens,
                              abundance=x)
    return syn.model_clumpy_3d(n=n, seed=seed, nside=c["nside"], n_q=c["n_q"], n_lev=c["n_lev"])


def _directions(nside):
    """HEALPix ring-scheme pixel centres (Gorski et al. 2005), [12 nside^2][3]."""
    d = []
    for i in range(1, 4 * nside):
        k = i if i < nside else (4 * nside - i if i > 3 * nside else nside)
        if nside <= i <= 3 * nside:
            z, s = 4.0 / 3.0 - 2.0 * i / (3.0 * nside), (i - nside + 1) % 2
        else:
            z, s = (1.0 - k * k / (3.0 * nside * nside)) * (1.0 if i < nside else -1.0), 1
        for j in range(1, 4 * k + 1):
            phi = math.pi / (2.0 * k) * (j - 0.5 * s)
            d.append((math.sqrt((1.0 - z) * (1.0 + z)) * math.cos(phi),
                      math.sqrt((1.0 - z) * (1.0 + z)) * math.sin(phi), z))
    return np.array(d)


def _batch_sizes(c):
    """Uneven sizes around c["n"], from half to one and a half times it."""
    return [int(c["n"] * (0.5 + (i + 0.5) / c["models"])) for i in range(c["models"])]


def _scatter_opacity(m):
    return 1e-16 * m.n_coll / m.n_coll.mean()   # a dust-like opacity, 1/m


def _channels(c):
    return np.linspace(-12e3, 12e3, c["n_q"])


def _ray(c):
    return 7 * c["nside"] ** 2 + 1


def _grad_rows(c, seed):
    """Rows as the corpus has them: (log n, log T, log |grad v|, log tau) and level
    fractions near a Boltzmann distribution."""
    rng = np.random.default_rng(seed)
    n = c["n"]
    X = np.stack([rng.uniform(13, 18, n), rng.uniform(1, 2, n), rng.uniform(-12, -9, n), rng.uniform(-3, 4, n)], 1)
    J = np.arange(c["n_lev"])
    e = -2.4 * J * (J + 1) / 10.0 ** X[:, 1:2] * (1.0 + 0.3 * rng.random((n, 1)))
    y = (2 * J + 1) * np.exp(e)
    return X.astype(np.float32), (y / y.sum(1, keepdims=True)).astype(np.float32)


class _State:
    pass


def _context(c, m, stream):
    ctx = mg.Context(precision=mg.MG_FP64 if c["fp64"] else mg.MG_MIXED, alo_band=c.get("band", 0))
    ctx.set_stream(stream.cuda_stream)
    ctx.load_model(m, dirs=_directions(c["nside"]))
    return ctx


def prepare(case, seed):
    s = _State()
    s.case = case
    if case["kind"] == "grad":
        s.X, s.Y = _grad_rows(case, seed)
        s.net = mg.MLP(case["n_lev"], seed=seed)
        s.net.set_normalisation(s.X.mean(0), np.maximum(s.X.std(0), 1e-3))
        return s
    s.stream = torch.cuda.Stream()
    s.stream.wait_stream(torch.cuda.current_stream())
    models = [_model(case, seed * 16 + i, n) for i, n in enumerate(_batch_sizes(case))] if case["kind"] == "batch" \
        else [_model(case, seed)]
    s.ctx = [_context(case, m, s.stream) for m in models]
    if case["kind"] != "snapshot":
        for ctx in s.ctx:
            ctx.trace_rays()
            ctx.init_populations()
    ctx, n = s.ctx[0], models[0].n
    if case["kind"] == "batch":
        s.batch = mg.Batch(s.ctx)
    s.pops = [torch.empty(c.n, c.n_lev, dtype=torch.float64, device="cuda") for c in s.ctx]
    s.rad = [torch.empty(n, ctx.n_lines, dtype=torch.float64, device="cuda") for _ in range(3)]
    if case["kind"] == "step":
        if case.get("scatter"):
            ctx.set_scattering(_scatter_opacity(models[0]), tol=1e-10, max_iter=200)
        s.start = torch.empty_like(s.pops[0])
        ctx.get_populations_dev(s.start.data_ptr())
        if case.get("tuned"):
            ctx.autotune(reps=1)
    if case["kind"] == "image":
        s.u = _channels(case)
        s.image = torch.empty(n, case["n_q"], dtype=torch.float64, device="cuda")
        s.xy = torch.empty(n, 2, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    return s


def _radiation_into(ctx, bufs):
    """J, L and J_eff into device buffers, by the C interface."""
    rc = ctx.lib.mg_get_radiation_dev(ctx.h, *[b.data_ptr() for b in bufs])
    assert rc == mg.MG_OK, rc


def run(state):
    s, c = state, state.case
    if c["kind"] == "grad":
        loss, grad = s.net.loss_grad(s.X, s.Y)
        return np.float32(loss), grad
    here = torch.cuda.current_stream()
    s.stream.wait_stream(here)
    ctx = s.ctx[0]
    out = {}
    with torch.cuda.stream(s.stream):
        if c["kind"] == "step":
            ctx.set_populations_dev(s.start.data_ptr())
            ctx.formal_solve()
            _radiation_into(ctx, s.rad)
            ctx.update_populations()
            ctx.get_populations_dev(s.pops[0].data_ptr())
            out = dict(rad=s.rad, pops=s.pops)
        elif c["kind"] == "ali":
            ctx.init_populations()
            ctx.iterate()
            ctx.get_populations_dev(s.pops[0].data_ptr())
            out = dict(pops=s.pops)
        elif c["kind"] == "batch":
            for x in s.ctx:
                x.init_populations()
            s.batch.iterate()
            for x, p in zip(s.ctx, s.pops):
                x.get_populations_dev(p.data_ptr())
            out = dict(pops=s.pops)
        elif c["kind"] == "snapshot":
            stats, _ = ctx.trace_rays()
            ctx.init_populations()
            ctx.formal_solve()
            _radiation_into(ctx, s.rad)
            out = dict(rad=s.rad)
        else:
            ctx.image_dev(_ray(c), 0, s.u, s.image.data_ptr(), s.xy.data_ptr())
            out = dict(image=[s.image])
        if not c["fp64"]:
            out = {k: [x.float() for x in v] for k, v in out.items()}
    here.wait_stream(s.stream)
    if c["kind"] == "snapshot":
        out["elements"], out["expanded"], out["longest"] = (stats[k] for k in ("n_elements", "n_expanded",
                                                                              "max_pair_len"))
    if c["kind"] == "image":
        out["xy"] = s.xy
    return out


# --------------------------------------------------------------- needed work
def work(case):
    c = case
    if c["kind"] == "grad":
        w = 4 * 128 + 2 * 128 * 128 + 128 * c["n_lev"]
        return {"bytes": 4.0 * (c["n"] * (4 + c["n_lev"]) + 2 * w), "flops": 6.0 * c["n"] * w}
    rays = 12 * c["nside"] ** 2
    n = sum(_batch_sizes(c)) if c["kind"] == "batch" else c["n"]
    one = n / c.get("models", 1)
    # traced cells and expanded points per half-ray, as the models have them
    cells = one / 2 if c["model"] == "sphere" else (0.64 if c["model"] == "cloud" else 0.7) * one ** (1.0 / 3.0)
    points = cells if c["model"] == "sphere" else cells + (115.0 if c["model"] == "cloud" else 20.0)
    lines = c["n_lev"] - 1
    if c["kind"] == "image":
        return {"bytes": n * (32.0 * cells + 16.0 * lines + 8.0 * c["n_q"]), "flops": 40.0 * n * 2 * points * c["n_q"]}
    passes = {"ali": 12, "batch": 8}.get(c["kind"], 15 if c.get("scatter") else 1)
    store = (24.0 if c["fp64"] else 16.0) * n * rays * cells
    traced = 25 * 12.0 * n * rays * cells if c["kind"] == "snapshot" else 0.0   # flops of the neighbour walk
    return {"bytes": passes * (store + 8.0 * n * (5 * lines + 2 * c["n_lev"])),
            "flops": traced + passes * (15.0 * n * rays * points * lines * c["n_q"] + n * c["n_lev"] ** 3)}


# --------------------------------------------------- the same in 64-bit torch
def _dev(x, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(x), dtype=dtype, device="cuda")


class _Fields:
    """Fields of a model on the GPU, its widths, LTE populations and line constants."""

    def __init__(self, m):
        sp = m.species
        self.m, self.n = m, m.n
        self.pos, self.vel = _dev(m.pos), _dev(m.vel)
        self.b = torch.sqrt(2.0 * KB * _dev(m.T) / sp.mass + _dev(m.v_turb) ** 2)
        self.nspec = _dev(m.n_spec)
        E, g = _dev(sp.E), _dev(sp.g)
        w = g * torch.exp(-E / (KB * _dev(m.T)[:, None]))
        self.pops = self.nspec[:, None] * w / w.sum(1, keepdim=True)
        up, lo = np.asarray(sp.up, int), np.asarray(sp.lo, int)
        self.up, self.lo = _dev(up, torch.long), _dev(lo, torch.long)
        nu = (sp.E[up] - sp.E[lo]) / H
        bul = sp.A * C ** 2 / (2 * H * nu ** 3)
        self.nu, self.A, self.bul, self.blu = _dev(nu), _dev(sp.A), _dev(bul), _dev(bul * sp.g[up] / sp.g[lo])
        pre = H * self.nu / (4 * math.pi)
        self.eta = pre * self.A * self.pops[:, self.up]
        self.chi = pre * (self.pops[:, self.lo] * self.blu - self.pops[:, self.up] * self.bul)


def _walks_cloud(f, dirs, o):
    """Cells, path lengths and velocities of the half-rays of origins o: [rays][steps]
    tensors padded with cell -1."""
    m = f.m
    if not hasattr(f, "nbr"):
        deg = np.diff(m.nbr_off)
        tab = np.full((m.n, deg.max()), -1, np.int64)
        row = np.repeat(np.arange(m.n), deg)
        tab[row, np.arange(len(row)) - np.repeat(m.nbr_off[:-1], deg)] = m.nbr_idx
        f.nbr, f.bdy = _dev(tab, torch.long), _dev(m.is_bdy, torch.bool)
    d = dirs.repeat(len(o), 1)
    oo = o.repeat_interleave(dirs.shape[0])
    x0, v0, cur, s = f.pos[oo], f.vel[oo], oo.clone(), torch.zeros(len(oo), dtype=torch.float64, device="cuda")
    alive = torch.ones(len(oo), dtype=torch.bool, device="cuda")
    cells, ds, v = [], [], []
    while bool(alive.any()):
        cand = f.nbr[cur]
        dx = f.pos[cand.clamp(min=0)] - x0[:, None]
        sc = (dx * d[:, None]).sum(-1)
        d2 = ((dx - sc[..., None] * d[:, None]) ** 2).sum(-1)
        d2 = torch.where((cand >= 0) & (sc > s[:, None]), d2, torch.inf)
        best, k = d2.min(1)
        alive = alive & torch.isfinite(best)
        nxt = cand.gather(1, k[:, None])[:, 0]
        ns = sc.gather(1, k[:, None])[:, 0]
        cells.append(torch.where(alive, nxt, -1))
        ds.append(ns - s)
        v.append(((f.vel[nxt.clamp(min=0)] - v0) * d).sum(-1))
        cur, s = torch.where(alive, nxt, cur), torch.where(alive, ns, s)
        alive = alive & ~f.bdy[cur]
    return torch.stack(cells, 1), torch.stack(ds, 1), torch.stack(v, 1)


def _walks_sphere(f, dirs, o):
    """The same for shells at rest around an empty core."""
    r = f.m.pos[:, 2]
    rows = []
    for i in o.tolist():
        for mu in dirs[:, 2].tolist():
            p2, cells, s = r[i] ** 2 * (1 - mu * mu), [], [0.0]
            j = i + 1
            if mu < 0:
                k = i - 1
                while k >= 0 and r[k] ** 2 > p2:
                    cells.append(k)
                    s.append(-r[i] * mu - math.sqrt(r[k] ** 2 - p2))
                    k -= 1
                j = k + 1
            core = mu < 0 and j == 0
            for k in range(j, len(r)):
                cells.append(k)
                s.append(-r[i] * mu + math.sqrt(max(r[k] ** 2 - p2, 0.0)))
            ds = np.diff(s)
            if core:
                ds[i] = 0.0
            rows.append((cells, ds))
    w = max(1, max(len(c) for c, _ in rows))
    cells, ds = np.full((len(rows), w), -1, np.int64), np.zeros((len(rows), w))
    for k, (c, d) in enumerate(rows):
        cells[k, :len(c)], ds[k, :len(c)] = c, d
    cells, ds = _dev(cells, torch.long), _dev(ds)
    return cells, ds, torch.zeros_like(ds)


def _points(f, dirs, o):
    """Points of the half-rays of origins o after velocity-step insertion, from the origin
    outwards: path length, velocity, width, the two cells and the weight on the second,
    [len(o)][rays][points], and the number of points [len(o)][rays]."""
    walk = _walks_sphere if f.m.geometry == mg.MG_GEOM_SPHERICAL_1D else _walks_cloud
    cells, ds, v = walk(f, dirs, o)
    R = dirs.shape[0]
    oo = o.repeat_interleave(R)
    ok = cells >= 0
    cb = cells.clamp(min=0)
    ca = torch.cat([oo[:, None], cb[:, :-1]], 1)
    va = torch.cat([torch.zeros_like(v[:, :1]), v[:, :-1]], 1)
    dv, lim = (v - va).abs(), DSHIFT * torch.minimum(f.b[ca], f.b[cb])
    sub = torch.where(dv > lim, torch.ceil(dv / lim), torch.ones_like(dv))
    sub = torch.where(ok, sub, torch.zeros_like(sub)).long()
    end = sub.cumsum(1)
    K = end[:, -1]
    x = torch.arange(int(K.max()) if len(K) else 0, device="cuda").expand(len(oo), -1).contiguous()
    e = torch.searchsorted(end, x, right=True).clamp(max=cells.shape[1] - 1)
    n_sub = sub.gather(1, e).clamp(min=1)
    w = (x - (end - sub).gather(1, e) + 1).double() / n_sub
    a, b = ca.gather(1, e), cb.gather(1, e)
    shape = (len(o), R, x.shape[1])
    return dict(ds=(ds.gather(1, e) / n_sub).view(shape), v=((1 - w) * va.gather(1, e) + w * v.gather(1, e)).view(shape),
                b=((1 - w) * f.b[a] + w * f.b[b]).view(shape), a=a.view(shape), c=b.view(shape), w=w.view(shape),
                K=K.view(shape[:2]))


def _planck(nu):
    return 2.0 * H * nu ** 3 / C ** 2 / torch.expm1(H * nu / (KB * T_CMB))


def _radiation(f, c, most=2e7):
    """J, L and J_eff of all points: per half-ray the two-ended elimination of the
    second-order transfer equation, one row at a time over all bins."""
    dirs = _dev(_directions(c["nside"]))
    anti = torch.cdist(dirs, -dirs).argmin(1)
    R = len(dirs)
    x, wq = np.polynomial.hermite.hermgauss(c["n_q"])
    roots, wq = _dev(x), _dev(wq / math.sqrt(math.pi))
    L = len(f.nu)
    out = [torch.empty(f.n, L, dtype=torch.float64, device="cuda") for _ in range(3)]
    step = max(1, int(most / (R * L * c["n_q"])))
    for o0 in range(0, f.n, step):
        o = torch.arange(o0, min(f.n, o0 + step), device="cuda")
        p = _points(f, dirs, o)
        aq = (f.b[o][:, None] * roots)[:, None, None, :]                    # [o][1][1][q]

        def at(b, v, eta, chi):
            """Floored opacity, source and line opacity at points of one index."""
            phi = torch.exp(-((aq * (1 - v / C) - v) / b) ** 2) * (C / (f.nu[:, None] * b * math.sqrt(math.pi)))
            own = chi * phi
            chi = own.clamp(min=CHI_MIN)
            return chi, eta * phi / chi, own

        nu_o = f.nu[:, None] * (1 + aq / C)
        I_o = _planck(nu_o)
        shape = (len(o), R, L, c["n_q"])
        F = torch.ones(shape, dtype=torch.float64, device="cuda")            # Phi iota
        psi = I_o.expand(shape).clone()
        dtp, chip, Sp = torch.zeros_like(F), torch.zeros_like(F), torch.zeros_like(F)
        own = None
        for k in range(p["ds"].shape[2] - 1, -2, -1):
            if k >= 0:
                a, b, w = p["a"][..., k], p["c"][..., k], p["w"][..., k][..., None, None]
                v, bb = p["v"][..., k][..., None, None], p["b"][..., k][..., None, None]
                eta = (1 - w) * f.eta[a][..., None] + w * f.eta[b][..., None]
                chi = (1 - w) * f.chi[a][..., None] + w * f.chi[b][..., None]
                chi, S, _ = at(bb, v, eta, chi)
            else:
                zero = torch.zeros(len(o), 1, 1, 1, dtype=torch.float64, device="cuda")
                chi, S, own = at(f.b[o][:, None, None, None], zero, f.eta[o][:, None, :, None],
                                 f.chi[o][:, None, :, None])
            K = p["K"][..., None, None]
            if k + 1 < p["ds"].shape[2]:
                inner = K > k + 1
                dt = (0.5 * (chip + chi) * p["ds"][..., k + 1][..., None, None]).clamp(min=DTAU_MIN)
                t = 0.5 * (dtp + dt)
                Phi = t + F
                iota = 1.0 / (1.0 + dt * Phi)
                F = torch.where(inner, Phi * iota, F)
                psi = torch.where(inner, (t * Sp + psi) * iota, psi)
                dtp = torch.where(inner, dt, dtp)
            if k >= 0:
                last = K == k + 1
                if bool(last.any()):
                    psi = torch.where(last, _planck(nu_o * (1 - v / C)), psi)
                chip, Sp = chi.expand(shape), S.expand(shape)
        d = dtp + dtp[:, anti]
        sig = torch.where(d > 0, 2.0 / d, torch.zeros_like(d))
        pi2, ps = sig * (F + F[:, anti]), sig * (psi + psi[:, anti])
        lam = torch.where(d > 0, 1.0 / (1.0 + pi2), torch.zeros_like(d))
        uml = torch.where(d > 0, ps * lam, psi)
        u = uml + S * lam
        share = own / chi
        for dst, val in zip(out, (u, lam * share, uml + lam * S * (1 - share))):
            dst[o] = (val * wq).sum(-1).mean(1)
    return out


def _rates(f, J_eff, one_minus_L):
    """Rate matrix [cell][from][to] of the statistical equilibrium."""
    sp, m = f.m.species, f.m
    n = sp.n_lev
    q = torch.zeros(f.n, n, n, dtype=torch.float64, device="cuda")
    for l, (u, d) in enumerate(zip(sp.up.tolist(), sp.lo.tolist())):
        q[:, u, d] += f.A[l] * one_minus_L[:, l] + f.bul[l] * J_eff[:, l]
        q[:, d, u] += f.blu[l] * J_eff[:, l]
    pr = 0
    for i in range(1, n):
        for j in range(i):
            k = _dev(np.interp(m.T, sp.T_grid, sp.K_down[pr]) * m.n_coll)
            q[:, i, j] += k
            q[:, j, i] += k * (sp.g[i] / sp.g[j]) * torch.exp(-(sp.E[i] - sp.E[j]) / (KB * _dev(m.T)))
            pr += 1
    return q


def _equilibrium(f, q):
    """Stationary populations by state reduction (Grassmann, Taksar & Heyman 1985)."""
    n = q.shape[1]
    out = [None] * n
    for k in range(n - 1, 0, -1):
        out[k] = q[:, k, :k].sum(1)
        q[:, :k, :k] += (q[:, :k, k] / out[k][:, None])[..., None] * q[:, k, None, :k]
    pi = torch.ones(f.n, n, dtype=torch.float64, device="cuda")
    for k in range(1, n):
        pi[:, k] = (pi[:, :k] * q[:, :k, k]).sum(1) / out[k]
    return f.nspec[:, None] * pi / pi.sum(1, keepdim=True)


def _image(f, c):
    """The intensity leaving along the ray through each point: linear source in tau."""
    dirs = _directions(c["nside"])
    n = dirs[_ray(c)]
    both = _dev(np.stack([-n, n]))
    u, nd = _dev(_channels(c)), _dev(n)
    I_all = torch.empty(f.n, c["n_q"], dtype=torch.float64, device="cuda")
    nu = float(f.nu[0])
    for o0 in range(0, f.n, 2048):
        o = torch.arange(o0, min(f.n, o0 + 2048), device="cuda")
        p = _points(f, both, o)
        vo = (f.vel[o] * nd).sum(1)[:, None]
        I = torch.zeros(len(o), c["n_q"], dtype=torch.float64, device="cuda")
        chip, Sp = torch.zeros_like(I), torch.zeros_like(I)
        begun = torch.zeros(len(o), 1, dtype=torch.bool, device="cuda")
        dsp = torch.zeros(len(o), 1, dtype=torch.float64, device="cuda")
        N = p["ds"].shape[2]
        for k in list(range(N - 1, -1, -1)) + [-1] + [N + i for i in range(N)]:
            if k == -1:
                on = torch.ones_like(begun)
                w, b, eta, chi = vo, f.b[o][:, None], f.eta[o, 0][:, None], f.chi[o, 0][:, None]
                ds = dsp
            else:
                h, i = (0, k) if k < N else (1, k - N)
                on = (p["K"][:, h] > i)[:, None]
                w = vo + (-1 if h == 0 else 1) * p["v"][:, h, i][:, None]
                b, wt = p["b"][:, h, i][:, None], p["w"][:, h, i]
                a, cc = p["a"][:, h, i], p["c"][:, h, i]
                eta = ((1 - wt) * f.eta[a, 0] + wt * f.eta[cc, 0])[:, None]
                chi = ((1 - wt) * f.chi[a, 0] + wt * f.chi[cc, 0])[:, None]
                ds = dsp if h == 0 else p["ds"][:, h, i][:, None]
            phi = torch.exp(-((u - w * (1 + u / C)) / b) ** 2) * (C / (nu * b * math.sqrt(math.pi)))
            chi = (chi * phi).clamp(min=CHI_MIN)
            S = eta * phi / chi
            dt = (0.5 * (chip + chi) * ds).clamp(min=DTAU_MIN)
            e = torch.exp(-dt)
            al = -torch.expm1(-dt) / dt
            wb = torch.where(dt < 1e-3, dt * (0.5 - dt * (1 / 6 - dt * (1 / 24 - dt / 120))), 1 - al)
            wa = torch.where(dt < 1e-3, dt * (0.5 - dt * (1 / 3 - dt * (1 / 8 - dt / 30))), al - e)
            new = torch.where(begun, e * I + wa * Sp + wb * S, _planck(nu * (1 + u / C) * (1 - w / C)))
            I = torch.where(on, new, I)
            chip, Sp = torch.where(on, chi, chip), torch.where(on, S, Sp)
            if k >= 0 and k < N:
                dsp = torch.where(on, p["ds"][:, 0, k][:, None], dsp)
            begun = begun | on
        I_all[o] = I
    ax = np.array([1.0, 0, 0]) if abs(n[2]) >= 0.9 else np.array([0, 0, 1.0])
    e1 = np.cross(ax, n)
    e1 /= np.linalg.norm(e1)
    return dict(image=[I_all], xy=f.pos @ _dev(np.stack([e1, np.cross(n, e1)], 1)))


def _grad(case, seed):
    X, Y = _grad_rows(case, seed)
    net = mg.MLP(case["n_lev"], seed=seed)   # the initial weights only
    theta = _dev(net.get_params()).requires_grad_()
    net.close()
    mean, std = X.mean(0), np.maximum(X.std(0), 1e-3)
    h, at = (_dev(X) - _dev(mean)) / _dev(std), 0
    width = [4, 128, 128, 128, case["n_lev"]]
    for i, (a, b) in enumerate(zip(width[:-1], width[1:])):
        W, bias = theta[at:at + a * b].view(a, b), theta[at + a * b:at + a * b + b]
        at += a * b + b
        h = h @ W + bias
        h = torch.relu(h) if i < 3 else torch.log_softmax(h, 1)
    Y = _dev(Y)
    on = Y >= 1e-12
    loss = ((h - torch.log(Y.clamp(min=1e-30))) ** 2)[on].mean()
    loss.backward()
    return np.float64(loss.item()), theta.grad


def exact(case, seed):
    c = case
    if c["kind"] == "grad":
        return _grad(c, seed)
    if c["kind"] in ("ali", "batch") or c.get("scatter"):
        return None   # many formal solves
    f = _Fields(_model(c, seed))
    if c["kind"] == "image":
        return _image(f, c)
    if c["n"] * 12 * c["nside"] ** 2 * len(f.nu) * c["n_q"] * (1 if c["model"] == "sphere" else 3) > 1e9:
        return None   # over 20 s
    J, L, E = _radiation(f, c)
    if c["kind"] == "snapshot":
        return dict(rad=[J, L, E])
    pops = None if c.get("band") else _equilibrium(f, _rates(f, E, 1.0 - L))
    return dict(rad=[J, L, E], pops=[pops])
