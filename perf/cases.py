"""What the performance of this framework is measured on: the calls its users
make, with inputs drawn from a seed.

The kinds of work, each through the public entry points of the package:

* ``trace``: ray bundles through an isolated halo or a replicated box on
  device arrays (rt3d_trace_device), in mixed precision or all in FP64;
* ``call``: the same through the host call (rt3d_trace) of a small program;
* ``survey``: a new particle set loaded, traced and binned, host buffers
  throughout (rt3d_load_particles, rt3d_trace, rt3d_histogram);
* ``cones``: many uneven light cones in one batched call (rt3d_trace_batch);
* ``grid``: the paper's grid force path, node grid built and traced
  (rt3d_load_grid, rt3d_trace_device);
* ``planes``: the multiple lens-plane comparison system
  (rt3d_multiplane_device);
* ``born``: convergence and shear maps in the Born approximation (rt3d_born);
* ``mupdf``: the magnification PDF of a finished map (rt3d_histogram_device).

Sizes come from the workloads of ``inputs/generators.py``, ``bench.py`` and the
tests, with fewer bundles or steps where a whole workload takes minutes; the
contexts are created with the library's default options.  ``exact`` is the
method written out in 64-bit torch, without this repository's code.
"""
import math

import numpy as np
import torch

import paper_1110_4894_gb300 as P

OM, OL, H = 0.3, 0.7, 0.7  # the cosmology of every workload
MU_G = 1.32712440018e20 / 299792458.0 ** 2 / 3.0856775814913673e22  # G Msun / c^2 in Mpc
H0 = 100.0 * H / 299792.458
QUANTUM = 2.0 ** -22  # particle coordinates are multiples of this many Mpc
ARCSEC = math.radians(1.0 / 3600.0)
MAX_EXTRA = 16
SUMMARY = ("mu", "kappa", "gamma1", "gamma2", "omega")


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # one point mass, all FP64, the Schwarzschild tests of Sec. 4.1: 66
        # bundles (an odd number of warps), a thousand steps of almost no work
        dict(name="point_lens", kind="trace", source="point", fp64=True, particles=1, bundles=66, ring=4, steps=1000),
        # the smallest call a program makes: a few bundles through a coarse halo
        dict(name="halo_few", kind="call", source="halo", fp64=False, particles=5000, bundles=4, ring=4, steps=200),
        # the NFW tests of Sec. 4.2 (100 000 particles, 64 x 64 bundles)
        dict(name="halo", kind="trace", source="halo", fp64=False, particles=100000, bundles=4096, ring=4, steps=30),
        # the paper's bundle of 8 rays; masses and softenings of their own per
        # particle, as an adaptive simulation writes them; ragged sizes
        dict(name="halo_ring8", kind="trace", source="halo", fp64=False, particles=30011, bundles=1111, ring=8,
             steps=100, varied=True),
        # the all-FP64 path on a halo, which the mixed results are checked with
        dict(name="halo_fp64", kind="trace", source="halo", fp64=True, particles=20000, bundles=256, ring=4, steps=16),
        # the 2^21-particle box replicated to z = 0.5 with the mean density
        # removed: the largest share of real running time
        dict(name="box", kind="trace", source="box", fp64=False, particles=2097152, bundles=768, ring=4, steps=48),
        # a snapshot read, traced and binned once
        dict(name="survey", kind="survey", source="box", fp64=False, particles=1048576, bundles=128, ring=4, steps=48),
        # many lines of sight of very different size in one launch
        dict(name="cones", kind="cones", cones=48, most=200000, ring=4, steps=16),
        # the paper's own force path: CIC, FFT, splines; then a trace on it
        dict(name="grid", kind="grid", source="halo", fp64=False, particles=100000, nodes=128, window=2, bundles=4096,
             ring=4, steps=500),
        # lens planes, two per replica
        dict(name="planes", kind="planes", source="box", fp64=False, particles=524288, bundles=4096, ring=4, slices=2),
        # Born maps of the halo
        dict(name="born", kind="born", source="halo", fp64=False, particles=100000, bundles=2048, steps=500),
        # the magnification PDF of a 1024 x 1024 map
        dict(name="mupdf", kind="mupdf", values=1048576, bins=200),
    ]


# no drawn case has more pair interactions (FP64 ones counted as 64) than the box
MOST_PAIRS = 4 * 48 * 768 * 5 * 2097152


def draw(rng):
    def span(lo, hi):  # log-uniform whole number
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(("trace", "trace", "trace", "call", "survey", "cones", "grid", "planes", "born", "mupdf"))
    if kind == "mupdf":
        return dict(kind=kind, values=span(20000, 1 << 20), bins=span(50, 400))
    if kind == "cones":
        return dict(kind=kind, cones=span(6, 48), most=span(10000, 200000), ring=rng.choice((4, 4, 8)),
                    steps=span(8, 24))
    if kind == "grid":
        return dict(kind=kind, source="halo", fp64=rng.random() < 0.25, particles=span(2000, 200000),
                    nodes=span(24, 128), window=rng.choice((1, 2, 2, 3, 4)), bundles=span(64, 8192),
                    ring=rng.choice((4, 4, 8)), steps=span(50, 500))
    if kind == "planes":
        return dict(kind=kind, source="box", fp64=False, particles=span(1 << 16, 1 << 20), bundles=span(256, 4096),
                    ring=rng.choice((4, 4, 8, 6)), slices=rng.choice((1, 1, 2, 3, 4)))
    if kind == "born":
        return dict(kind=kind, source="halo", fp64=False, particles=span(3000, 150000), bundles=span(64, 4096),
                    steps=span(100, 600))
    if kind == "survey":
        return dict(kind=kind, source="box", fp64=False, particles=span(1 << 16, 1 << 20), bundles=span(32, 256),
                    ring=4, steps=span(24, 64))
    if kind == "call":
        return dict(kind=kind, source="halo", fp64=False, particles=span(1000, 20000), bundles=span(1, 64),
                    ring=rng.choice((4, 4, 8)), steps=span(50, 300))
    source = rng.choice(("halo", "halo", "halo", "box", "box", "point"))
    case = dict(kind="trace", source=source, fp64=source == "point" or rng.random() < 0.2,
                ring=rng.choice((4, 4, 4, 8, 8, 3, 5, 6)))
    if source == "point":
        case.update(particles=1, bundles=span(16, 512), steps=span(200, 1000))
    elif source == "halo":
        case.update(particles=span(1000, 200000), bundles=span(16, 8192), steps=span(16, 200),
                    varied=rng.random() < 0.3)
    else:
        case.update(particles=span(1 << 17, 1 << 21), bundles=span(64, 1024), steps=span(32, 96))
    while _pairs(case) * (64 if case["fp64"] else 1) > MOST_PAIRS:
        for k, least in (("bundles", 16), ("steps", 16), ("particles", 1000)):
            case[k] = max(least, int(case[k] * 0.83)) if case[k] > 1 else 1
    return case


def _pairs(c):
    """ray-particle pairs of one pass (each at one RK4 stage)"""
    return 4 * c["steps"] * c["bundles"] * (1 + c["ring"]) * c["particles"]


def work(case):
    c, kind = case, case["kind"]
    if kind == "mupdf":  # mu and flags in, bins out; a logarithm, a division and the moments per value
        return dict(bytes=16 * c["values"] + 16 * c["bins"] + 64, flops=40 * c["values"])
    if kind == "cones":
        n, rays, pairs = 0, 0, 0
        for k in _cone_sizes(c, 0):
            n += k["particles"]
            rays += k["bundles"] * (1 + c["ring"])
            pairs += 4 * c["steps"] * k["bundles"] * (1 + c["ring"]) * k["particles"]
        return dict(bytes=16 * n + 64 * rays, flops=20 * pairs)
    if kind == "born":  # three Hessian combinations per pair
        return dict(bytes=16 * c["particles"] + 40 * c["bundles"],
                    flops=18 * (c["steps"] + 1) * c["bundles"] * c["particles"])
    rays = c["bundles"] * (1 + c["ring"])
    out = 64 * rays + 64 * c["bundles"]
    if kind == "planes":  # each particle up to the source is on one plane
        return dict(bytes=16 * c["particles"] + out, flops=12 * rays * c["particles"] * 1888.0 / _box_side(c))
    if kind == "grid":  # the interpolation and the integrator per ray and stage, nine transforms of the padded grid
        p3 = 8 * c["nodes"] ** 3
        return dict(bytes=32 * c["particles"] + out + 32 * c["nodes"] ** 3,
                    flops=4 * c["steps"] * rays * (32 * (2 * c["window"]) ** 2 + 300) +
                    9 * 2.5 * p3 * math.log2(p3))
    return dict(bytes=(32 if kind == "survey" else 16) * c["particles"] + out, flops=20 * _pairs(c))


# ---------------------------------------------------------------------------
# background cosmology (flat LCDM, 64-bit numpy)
# ---------------------------------------------------------------------------
_X64, _W64 = np.polynomial.legendre.leggauss(64)
_X8, _W8 = np.polynomial.legendre.leggauss(8)


def _chi(z):
    z = np.asarray(z, np.float64)
    u = 1.0 + 0.5 * z[..., None] * (_X64 + 1.0)
    return (_W64 / np.sqrt(OM * u ** 3 + OL)).sum(-1) * 0.5 * z / H0


def _redshift(chi):
    chi = np.asarray(chi, np.float64)
    z = chi * H0
    for _ in range(7):
        z = z - (_chi(z) - chi) * H0 * np.sqrt(OM * (1.0 + z) ** 3 + OL)
    return z


def _nodes(kind, n, chi_s, chi_l, s):
    k = np.arange(n + 1) / n
    if kind == P.SCHED_UNIFORM:
        x = chi_s * k
    else:
        u0, u1 = math.asinh(-chi_l / s), math.asinh((chi_s - chi_l) / s)
        x = chi_l + s * np.sinh(u0 + (u1 - u0) * k)
        x[0], x[-1] = 0.0, chi_s
    return x


def _steps(x):
    """the affine steps int a^2 dchi between the nodes x"""
    e = np.concatenate([x[:-1, None] + (x[1:] - x[:-1])[:, None] * np.arange(4) / 4, x[1:, None]], axis=1)
    w = e[:, 1:] - e[:, :-1]
    p = e[:, :-1, None] + 0.5 * w[..., None] * (_X8 + 1.0)
    return ((_W8 * (1.0 + _redshift(p)) ** -2).sum(-1) * 0.5 * w).sum(-1)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _rng(seed, *purpose):
    return np.random.Generator(np.random.PCG64(np.random.SeedSequence([int(seed), *purpose])))


def _quantize(x):
    return np.round(x / QUANTUM) * QUANTUM


_NFW_X = np.concatenate([[0.0], np.geomspace(1e-4, 60.0, 4000)])
_NFW_M = np.log1p(_NFW_X) - _NFW_X / (1.0 + _NFW_X)


def _nfw(g, conc, trunc=2.0):
    """offsets in units of r200 of one particle of an NFW halo per entry of conc"""
    x_t = trunc * conc
    m = g.random(conc.shape[0]) * (np.log1p(x_t) - x_t / (1.0 + x_t))
    r = np.interp(m, _NFW_M, _NFW_X) / conc
    ct, ph = g.uniform(-1.0, 1.0, r.shape[0]), g.uniform(0.0, 2.0 * math.pi, r.shape[0])
    st = np.sqrt(1.0 - ct * ct)
    return np.stack([r * st * np.cos(ph), r * st * np.sin(ph), r * ct], axis=1)


def _r200(mass, z):
    return (MU_G * mass / (100.0 * H0 * H0 * (OM * (1 + z) ** 3 + OL))) ** (1.0 / 3.0)


def _square(g, lo, hi, n):
    """n bundle centres of a square grid, tile by tile of 8 x 8 so that
    neighbours in the list are neighbours on the sky; each a little off its
    grid point, so that another seed is another map"""
    side = int(math.ceil(math.sqrt(n)))
    t = np.linspace(lo, hi, side) if side > 1 else np.array([0.5 * (lo + hi)])
    i, j = (v.ravel() for v in np.meshgrid(np.arange(side), np.arange(side), indexing="ij"))
    order = np.lexsort((j % 8, i % 8, j // 8, i // 8))[:n]
    th = np.stack([t[i[order]], t[j[order]]], axis=1)
    return th + g.uniform(-0.2, 0.2, th.shape) * (hi - lo) / side


def _box_side(c):
    """the box length: 100/h Mpc for 2^21 particles, the same mean density for fewer"""
    L = 100.0 / H * (c["particles"] / 2097152.0) ** (1.0 / 3.0)
    return round(L / (2 * QUANTUM)) * 2 * QUANTUM


def _box(seed, n, L):
    """a periodic box: half the particles uniform, half in NFW halos with dN/dM ~ M^-1.9"""
    g = _rng(seed, 1)
    halos = max(1, int(round(3000 * n / 2097152.0)))
    u = g.random(halos)
    M = (1e11 ** -0.9 + u * (1e15 ** -0.9 - 1e11 ** -0.9)) ** (-1.0 / 0.9)
    n_h = n // 2
    count = np.floor(M / M.sum() * n_h).astype(np.int64)
    count[np.argmax(M)] += n_h - count.sum()
    who = np.repeat(np.arange(halos), count)
    pos = g.random((halos, 3))[who] * L + _nfw(g, (5.0 * (M / 1e14) ** -0.1)[who]) * _r200(M, 0.0)[who, None]
    pos = np.mod(_quantize(np.concatenate([pos, g.random((n - n_h, 3)) * L])), L)
    pos[pos >= L] = 0.0
    return pos, np.full(n, M.sum() / n_h)


def _replicas(seed, count, L):
    g = _rng(seed, 2)
    rot = np.zeros((count, 3, 3), np.int32)
    for r in rot:
        r[np.arange(3), g.permutation(3)] = g.choice((-1, 1), 3)
        if np.linalg.det(r) < 0:
            r[0] *= -1
    shift = np.mod(_quantize(g.random((count, 3)) * L), L)
    return rot, shift


def _inputs(case, seed):
    """the arrays and options of one case, as a program has them before the call"""
    c, g = case, _rng(seed, 3)
    if c["kind"] == "mupdf":
        n = c["values"]
        out = np.zeros((n, 6))
        k = np.abs(g.standard_normal(n)) ** 1.5 * 0.03 - 0.02  # skewed, with a tail of strong lensing
        out[:, 1] = k
        out[:, 2:4] = 0.02 * g.standard_normal((n, 2))
        out[:, 0] = 1.0 / ((1.0 - k) ** 2 - out[:, 2] ** 2 - out[:, 3] ** 2)
        bad = g.random(n) < 1e-3
        out[bad, 0] = np.nan
        out[:, 5] = np.where(bad, 2.0, np.where(out[:, 0] < 0, 4.0, 0.0))
        return dict(bundles=out)
    if c["kind"] == "cones":
        return dict(cones=[_light_cone(k) for k in _cone_sizes(c, seed)], ring=c["ring"], theta_r=ARCSEC)
    z_s, z_l = 0.5, 0.25
    n, chi_l = c["particles"], float(_chi(z_l))
    d = dict(z_s=z_s, ring=c.get("ring", 4), theta_r=ARCSEC, steps=c.get("steps", 1), schedule=P.SCHED_ASINH,
             lens_chi=chi_l, replicated=False)
    if c["source"] == "point":
        M, chi_s = 1e12 * 10.0 ** g.uniform(-0.3, 0.3), float(_chi(z_s))
        th_E = math.sqrt(4 * MU_G * M * (1 + z_l) * (chi_s - chi_l) / (chi_l * chi_s))
        pos = _quantize(np.array([[0.0, 0.0, chi_l]]))
        x = np.linspace(0.5, 5.0, c["bundles"]) * th_E
        return dict(d, pos=pos, mass=np.array([M]), soft=0.0, theta=np.stack([x, np.zeros_like(x)], 1),
                    theta_r=1e-3 * th_E, lens_chi=float(pos[0, 2]), asinh_s=0.2 * th_E * chi_l)
    if c["source"] == "halo":
        r200 = float(_r200(1e14, z_l))
        pos = _quantize(_nfw(g, np.full(n, 5.0)) * r200 * (1 + z_l) + np.array([0.0, 0.0, chi_l]))
        mass, soft = np.full(n, 1e14 * 1.6 / n), 5e-3
        if c.get("varied"):
            mass, soft = mass * g.uniform(0.5, 2.0, n), 5e-3 * g.uniform(0.5, 3.0, n)
        lo, hi = (f * r200 * (1 + z_l) / chi_l / math.sqrt(2) for f in (0.05, 2.0))
        return dict(d, pos=pos, mass=mass, soft=soft, theta=_square(g, lo, hi, c["bundles"]), asinh_s=5e-3)
    L = _box_side(c)
    pos, mass = _box(seed, n, L)
    chi_s = float(_chi(z_s))
    count = int(math.ceil(chi_s / L)) + 1
    rot, shift = _replicas(seed, count, L)
    half = min(math.radians(1.95), 0.4 * L / chi_s)
    return dict(d, pos=pos, mass=mass, soft=0.016 / H, theta=_square(g, -half, half, c["bundles"]),
                schedule=P.SCHED_UNIFORM, lens_chi=0.0, asinh_s=1.0, replicated=True, L=L, rot=rot, shift=shift)


def _cone_sizes(c, seed):
    """sizes are the case's (the same for every seed), contents the seed's"""
    g = _rng(c["cones"], c["most"], 4)
    return [dict(particles=int(round(math.exp(g.uniform(math.log(1e3), math.log(c["most"]))))),
                 bundles=int(round(math.exp(g.uniform(math.log(128), math.log(1024))))),
                 z_s=float(g.uniform(0.3, 1.5)), steps=c["steps"], seed=int(seed) * 1000 + i)
            for i in range(c["cones"])]


def _light_cone(k):
    L = round(50.0 / H / (2 * QUANTUM)) * 2 * QUANTUM
    pos, mass = _box(k["seed"], k["particles"], L)
    chi_s = float(_chi(k["z_s"]))
    rot, shift = _replicas(k["seed"], int(math.ceil(chi_s / L)) + 1, L)
    half = (0.5 * L - 5.0 / H) / chi_s
    return dict(pos=pos, mass=mass, soft=0.016 / H, L=L, rot=rot, shift=shift, z_s=k["z_s"], steps=k["steps"],
                theta=_square(_rng(k["seed"], 5), -half, half, k["bundles"]))


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _load(ctx, field, d):
    kw = dict(replicated=True, box_length=d["L"], rot=d["rot"], shift=d["shift"], mean_subtract=True) \
        if "L" in d else {}
    ctx.load_particles(field, d["pos"], d["mass"], d["soft"], **kw)


def _options(d):
    return dict(n_ring=d["ring"], theta_r=d["theta_r"], schedule=d["schedule"], n_steps=d["steps"],
                lens_chi=d["lens_chi"], asinh_s=d["asinh_s"], max_extra=MAX_EXTRA)


def prepare(case, seed):
    kind, d = case["kind"], _inputs(case, seed)
    ctx = P.Context(0, precision=P.FP64 if case.get("fp64") else P.MIXED)
    ctx.set_cosmology(OM, OL, H)
    s = dict(kind=kind, case=case, ctx=ctx, inputs=d)
    if kind == "mupdf":
        s["bundles"] = torch.from_numpy(d["bundles"]).cuda()
        s["counts"], s["weights"] = (torch.empty(case["bins"], dtype=torch.int64, device="cuda") for _ in range(2))
        s["scalars"] = torch.empty(8, dtype=torch.float64, device="cuda")
    elif kind == "cones":
        for i, k in enumerate(d["cones"]):
            _load(ctx, i, k)
        s["cones"] = [dict(field_id=i, z_s=k["z_s"], theta=k["theta"], n_steps=k["steps"])
                      for i, k in enumerate(d["cones"])]
    elif kind == "grid":
        span = 2.2 * float(_r200(1e14, 0.25)) * 1.25
        s["lo"], s["spacing"] = (-span, -span, d["lens_chi"] - span), 2 * span / (case["nodes"] - 1)
    elif kind != "survey":
        _load(ctx, 0, d)
    if kind in ("trace", "grid", "planes"):
        nb, nr = d["theta"].shape[0], 1 + d["ring"]
        s["theta"] = torch.from_numpy(d["theta"]).cuda()
        s["bundles"] = torch.empty((nb, 6), dtype=torch.float64, device="cuda")
        s["rays"] = torch.empty((nb, nr, 8), dtype=torch.float64, device="cuda")
    return s


def _catalogue(r):
    """the bundles of a host result as one table (mu, kappa, gamma1, gamma2, omega) and their flags"""
    return np.stack([r[k] for k in SUMMARY], axis=1), r["flags"]


def run(state):
    s, ctx, d, kind = state, state["ctx"], state["inputs"], state["kind"]
    stream = torch.cuda.current_stream().cuda_stream
    if kind == "mupdf":
        ctx.histogram_device(stream, s["bundles"].shape[0], s["bundles"].data_ptr(), s["counts"].data_ptr(),
                             s["weights"].data_ptr(), s["scalars"].data_ptr(), bins=s["case"]["bins"])
        return [s["counts"], s["weights"], s["scalars"]]
    if kind == "cones":
        got = [_catalogue(r) for r in ctx.trace_batch(s["cones"], n_ring=d["ring"], theta_r=d["theta_r"],
                                                      max_extra=MAX_EXTRA)]
        return [np.concatenate([g[0] for g in got]), np.concatenate([g[1] for g in got])]
    if kind == "call":
        return list(_catalogue(ctx.trace(0, d["z_s"], d["theta"], **_options(d))))
    if kind == "survey":
        _load(ctx, 0, d)
        r = ctx.trace(0, d["z_s"], d["theta"], **_options(d))
        counts, weights, _ = ctx.histogram(r["mu"], r["flags"])
        return [*_catalogue(r), counts.astype(np.int64), weights.astype(np.int64)]
    if kind == "born":
        return [ctx.born(0, d["z_s"], d["theta"], n_ring=4, theta_r=d["theta_r"], schedule=d["schedule"],
                         n_steps=d["steps"], lens_chi=d["lens_chi"], asinh_s=d["asinh_s"])]
    ptr = (s["theta"].data_ptr(), s["bundles"].data_ptr())
    if kind == "planes":
        ctx.multiplane_device(stream, 0, d["z_s"], s["theta"].shape[0], *ptr, slices=s["case"]["slices"],
                              d_ray_out=s["rays"].data_ptr(), n_ring=d["ring"], theta_r=d["theta_r"])
        return [s["bundles"], s["rays"]]
    if kind == "grid":
        ctx.load_grid(0, d["pos"], d["mass"], d["soft"], s["lo"], s["spacing"], s["case"]["nodes"],
                      n_int=s["case"]["window"])
    ctx.trace_device(stream, 0, d["z_s"], s["theta"].shape[0], *ptr, d_ray_out=s["rays"].data_ptr(), **_options(d))
    return [s["bundles"], s["rays"]]


# ---------------------------------------------------------------------------
# the same in 64 bits, written out in torch
# ---------------------------------------------------------------------------
_LONG = 2.5e11  # pairs beyond which a direct sum in torch takes too long


def exact(case, seed):
    kind = case["kind"]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if kind == "mupdf":
        return [None, None, _exact_moments(torch.from_numpy(_inputs(case, seed)["bundles"]).to(dev), case["bins"])]
    if kind == "cones" or (kind in ("trace", "call", "survey") and _pairs(case) > _LONG):
        return None
    d = _inputs(case, seed)
    if kind == "born":
        if (case["steps"] + 1) * case["bundles"] * case["particles"] > _LONG:
            return None
        return [_exact_born(d, dev)]
    if kind == "planes":
        if case["bundles"] * (1 + case["ring"]) * case["particles"] * 1888.0 / d["L"] > _LONG:
            return None
        return list(_exact_planes(d, case["slices"], dev))
    if kind == "grid":
        span = 2.2 * float(_r200(1e14, 0.25)) * 1.25
        field = _GridField(d, (-span, -span, d["lens_chi"] - span), 2 * span / (case["nodes"] - 1), case["nodes"],
                           case["window"], dev)
    else:
        field = _DirectField(d, dev)
    bundles, rays = _exact_trace(d, field, dev)
    if kind == "call":
        return [bundles[:, :5], None]
    if kind == "survey":
        return [bundles[:, :5], None, None, None]
    return [bundles, rays]


def _exact_moments(b, bins, mu_min=0.5, mu_max=5.0):
    mu, flags = b[:, 0], b[:, 5].to(torch.int64)
    use = ((flags & 3) == 0) & torch.isfinite(mu) & (mu != 0)
    v = mu[use].abs()
    k = torch.floor((torch.log10(v) - math.log10(mu_min)) / ((math.log10(mu_max) - math.log10(mu_min)) / bins))
    W = (1.0 / v).sum()
    mean = torch.ones_like(v).sum() / W
    spread = torch.sqrt((((v - mean) ** 2) / v).sum() / W)
    counts = [use.sum(), (k < 0).sum(), (k >= bins).sum(), (mu[use] < 0).sum(), (~use).sum()]
    return torch.stack([torch.as_tensor(x, dtype=torch.float64, device=b.device) for x in (*counts, W, mean, spread)])


def _prism(lo, hi, p):
    """I = int dV / |p - r'| over the prism and its gradient, (n, 4)"""
    out = torch.zeros((p.shape[0], 4), dtype=torch.float64, device=p.device)

    def log_term(u, rho, q):
        return torch.where(u >= 0, torch.log(torch.where(u >= 0, u + rho, torch.ones_like(u))),
                           torch.log(q / torch.where(u >= 0, torch.ones_like(u), rho - u)))

    for corner in range(8):
        x, y, z = ((hi[k] if corner >> k & 1 else lo[k]) - p[:, k] for k in range(3))
        rho = torch.sqrt(x * x + y * y + z * z)
        lx, ly, lz = log_term(x, rho, y * y + z * z), log_term(y, rho, x * x + z * z), log_term(z, rho, x * x + y * y)
        tx, ty, tz = torch.atan(y * z / (x * rho)), torch.atan(z * x / (y * rho)), torch.atan(x * y / (z * rho))
        sign = -1.0 if (3 - bin(corner).count("1")) & 1 else 1.0
        out[:, 0] += sign * (x * y * lz + y * z * lx + z * x * ly - 0.5 * (x * x * tx + y * y * ty + z * z * tz))
        out[:, 1] -= sign * (y * lz + z * ly - x * tx)
        out[:, 2] -= sign * (z * lx + x * lz - y * ty)
        out[:, 3] -= sign * (x * ly + y * lx - z * tz)
    return out


def _placed(d, pos, j):
    """the box's particles in replica j, world coordinates"""
    R = torch.as_tensor(d["rot"][j], dtype=torch.float64, device=pos.device)
    s = torch.as_tensor(d["shift"][j], dtype=torch.float64, device=pos.device)
    L = d["L"]
    w = torch.remainder((pos - 0.5 * L) @ R.T + 0.5 * L + s, L)
    return w + torch.tensor([-0.5 * L, -0.5 * L, j * L], dtype=torch.float64, device=pos.device)


class _DirectField:
    """phi and grad phi of softened particles by direct summation"""

    def __init__(self, d, dev):
        self.d = d
        self.pos = torch.as_tensor(d["pos"], device=dev)
        self.m = torch.as_tensor(d["mass"], device=dev) * MU_G
        self.e2 = torch.as_tensor(np.broadcast_to(np.asarray(d["soft"], np.float64) ** 2, d["mass"].shape).copy(),
                                  device=dev)

    def __call__(self, p, rep):
        if not self.d["replicated"]:
            return self._sum(p, self.pos)
        out = torch.empty((p.shape[0], 4), dtype=torch.float64, device=p.device)
        L, n = self.d["L"], self.pos.shape[0]
        rho = float(self.m.sum()) / L ** 3
        for j in torch.unique(rep).tolist():
            at = rep == j
            q = p[at]
            out[at] = self._sum(q, _placed(self.d, self.pos, j)) + \
                rho * _prism((-0.5 * L, -0.5 * L, j * L), (0.5 * L, 0.5 * L, (j + 1) * L), q)
        return out

    def _sum(self, p, pos):
        out = torch.zeros((p.shape[0], 4), dtype=torch.float64, device=p.device)
        chunk = max(1, (1 << 24) // p.shape[0])
        for a in range(0, pos.shape[0], chunk):
            q, m, e2 = pos[a:a + chunk], self.m[a:a + chunk], self.e2[a:a + chunk]
            x, y, z = (q[None, :, k] - p[:, None, k] for k in range(3))
            inv = torch.rsqrt(x * x + y * y + z * z + e2)
            w = m * inv
            out[:, 0] -= w.sum(1)
            w *= inv * inv
            for k, v in enumerate((x, y, z)):
                out[:, 1 + k] -= (w * v).sum(1)
        return out


def _natural(n, device):
    """the matrix that takes n unit-spaced values to the second derivatives of their natural cubic spline"""
    A, B = np.zeros((n, n)), np.zeros((n, n))
    A[0, 0] = A[-1, -1] = 1.0
    for i in range(1, n - 1):
        A[i, i - 1:i + 2], B[i, i - 1:i + 2] = (1.0, 4.0, 1.0), (6.0, -12.0, 6.0)
    return torch.as_tensor(np.linalg.solve(A, B), device=device)


class _GridField:
    """the grid path: cloud-in-cell masses, zero-padded convolution, splines"""

    def __init__(self, d, lo, h, n, window, dev):
        f8 = dict(dtype=torch.float64, device=dev)
        self.n, self.h, self.W, self.lo = n, h, 2 * window, torch.tensor(lo, **f8)
        u = (torch.as_tensor(d["pos"], device=dev) - self.lo) / h
        i, f = torch.floor(u).to(torch.int64), u - torch.floor(u)
        node = torch.zeros(n ** 3, **f8)
        for c in range(8):
            s = torch.tensor([c & 1, c >> 1 & 1, c >> 2 & 1], device=dev)
            at = i + s
            w = torch.where(s == 1, f, 1.0 - f).prod(1) * torch.as_tensor(d["mass"], device=dev)
            ok = ((at >= 0) & (at < n)).all(1)
            node.index_add_(0, ((at[:, 0] * n + at[:, 1]) * n + at[:, 2])[ok], w[ok])
        k = torch.arange(2 * n, **f8)
        k = torch.where(k < n, k, k - 2 * n) * h
        r2 = k[:, None, None] ** 2 + k[None, :, None] ** 2 + k[None, None, :] ** 2 + float(d["soft"]) ** 2
        inv = torch.where(r2 > 0, torch.rsqrt(r2), torch.zeros_like(r2))
        for x in range(3):
            inv.select(x, n).zero_()
        spec = torch.fft.rfftn(node.view(n, n, n), s=(2 * n,) * 3)
        kernels = [-MU_G * inv] + [MU_G * k.view([-1 if a == x else 1 for a in range(3)]) * inv ** 3 for x in range(3)]
        val = torch.stack([torch.fft.irfftn(spec * torch.fft.rfftn(q), s=(2 * n,) * 3)[:n, :n, :n] for q in kernels], -1)
        self.tab = torch.cat([val, torch.einsum("ij,abjf->abif", _natural(n, dev), val)], -1).view(-1, 8)
        self.second = _natural(self.W, dev)

    def _weights(self, u):
        W = self.W
        k = torch.floor(u).clamp(0, W - 2).to(torch.int64)
        A, B = (k + 1) - u, u - k
        c = torch.zeros((u.shape[0], W), dtype=torch.float64, device=u.device)
        c.scatter_(1, k[:, None], A[:, None])
        c.scatter_add_(1, k[:, None] + 1, B[:, None])
        return c + ((A ** 3 - A) / 6.0)[:, None] * self.second[k] + ((B ** 3 - B) / 6.0)[:, None] * self.second[k + 1]

    def __call__(self, p, rep):
        n, W = self.n, self.W
        u = (p - self.lo) / self.h
        inside = ((u >= 0) & (u <= n - 1)).all(1)
        out = torch.zeros((p.shape[0], 4), dtype=torch.float64, device=p.device)
        u = u[inside]
        if not u.shape[0]:
            return out
        s = (torch.floor(u).to(torch.int64) - W // 2 + 1).clamp(0, n - W)
        k3 = torch.floor(u[:, 2]).clamp(0, n - 2).to(torch.int64)
        B = u[:, 2] - k3
        A = 1.0 - B
        c1, c2 = self._weights(u[:, 0] - s[:, 0]), self._weights(u[:, 1] - s[:, 1])
        w = torch.arange(W, device=p.device)
        line = ((s[:, 0, None, None] + w[:, None]) * n + s[:, 1, None, None] + w) * n + k3[:, None, None]
        a, b = self.tab[line], self.tab[line + 1]
        A, B = A[:, None, None, None], B[:, None, None, None]
        v = A * a[..., :4] + B * b[..., :4] + ((A ** 3 - A) * a[..., 4:] + (B ** 3 - B) * b[..., 4:]) / 6.0
        out[inside] = torch.einsum("na,nb,nabf->nf", c1, c2, v)
        return out


def _ray_angles(d, dev):
    th = torch.as_tensor(d["theta"], device=dev)
    ang = 2.0 * math.pi * torch.arange(d["ring"], dtype=torch.float64, device=dev) / d["ring"]
    ring = d["theta_r"] * torch.stack([torch.cos(ang), torch.sin(ang)], 1)
    return torch.cat([th[:, None], th[:, None] + ring], 1)  # (bundles, rays, 2)


def _jacobian(th, y, chi_s, crossed):
    """(mu, kappa, gamma1, gamma2, omega, flags) from the rays' source positions"""
    b, t = (y[:, 1:, 1:3] - y[:, :1, 1:3]) / chi_s, th[:, 1:] - th[:, :1]
    A = torch.linalg.solve(t.transpose(1, 2) @ t, t.transpose(1, 2) @ b).transpose(1, 2)
    mu = 1.0 / (A[:, 0, 0] * A[:, 1, 1] - A[:, 0, 1] * A[:, 1, 0])
    flags = torch.where(mu < 0, 4.0, 0.0) + torch.where(crossed, 0.0, 1.0)
    return torch.stack([mu, 1.0 - 0.5 * (A[:, 0, 0] + A[:, 1, 1]), 0.5 * (A[:, 1, 1] - A[:, 0, 0]),
                        -0.5 * (A[:, 0, 1] + A[:, 1, 0]), 0.5 * (A[:, 0, 1] - A[:, 1, 0]), flags], 1)


def _exact_trace(d, field, dev):
    """null geodesics of every ray by RK4 to the plane x3 = chi_s"""
    chi_s = float(_chi(d["z_s"]))
    dl = _steps(_nodes(d["schedule"], d["steps"], chi_s, d["lens_chi"], d["asinh_s"]))
    th = _ray_angles(d, dev)
    nb, nr = th.shape[:2]
    t0 = 2.0 / (3.0 * H0 * math.sqrt(OL)) * math.asinh(math.sqrt(OL / OM))
    y = torch.zeros((nb, nr, 8), dtype=torch.float64, device=dev)
    y[..., 5:7], y[..., 7] = th, 1.0

    def gather(y):
        rep = None
        if d["replicated"]:
            rep = torch.floor(y[:, 0, 3] / d["L"]).clamp(0, len(d["rot"]) - 1).to(torch.int64)
            rep = rep[:, None].expand(nb, nr).reshape(-1)
        return field(y[..., 1:4].reshape(-1, 3), rep).view(nb, nr, 4)

    def scale(y):
        return (OM / OL * torch.sinh(1.5 * math.sqrt(OL) * H0 * (t0 - y[..., 0])) ** 2) ** (1.0 / 3.0)

    def slope(y, F):
        a = scale(y)
        ad = -a * H0 * torch.sqrt(OM / a ** 3 + OL)
        phi, g, T, v = F[..., 0], F[..., 1:], y[..., 4], y[..., 5:]
        gv, v2 = (g * v).sum(-1), (v * v).sum(-1)
        dT = ad * phi / a ** 2 * T * T - 2.0 * gv * T / a - ad * (a + phi) * v2
        dv = -g * (T * T / a ** 3)[..., None] - (2.0 * ad * (a + phi) / a ** 2 * T)[..., None] * v - \
            (g * v2[..., None] - 2.0 * v * gv[..., None]) / a[..., None]
        return torch.cat([T[..., None], v, dT[..., None], dv], -1)

    fin, done = torch.zeros_like(y), torch.zeros((nb, nr), dtype=torch.bool, device=dev)
    for step in range(d["steps"] + MAX_EXTRA):
        if step >= d["steps"] and bool(done.all()):
            break
        h = float(dl[min(step, d["steps"] - 1)])
        F = gather(y)
        if step == 0:  # null condition at the observer
            a, vn = scale(y), y[..., 5:].norm(dim=-1)
            y[..., 4] = a * vn * torch.sqrt((1.0 - 2.0 * F[..., 0] / a) / (1.0 + 2.0 * F[..., 0] / a))
        k1 = slope(y, F)
        k2 = slope(y + 0.5 * h * k1, gather(y + 0.5 * h * k1))
        k3 = slope(y + 0.5 * h * k2, gather(y + 0.5 * h * k2))
        k4 = slope(y + h * k3, gather(y + h * k3))
        new = y + h / 6.0 * (k1 + 2.0 * k2 + 2.0 * k3 + k4)
        now = ~done & (new[..., 3] >= chi_s)
        s = (chi_s - y[..., 3]) / (new[..., 3] - y[..., 3])
        fin = torch.where(now[..., None], y + s[..., None] * (new - y), fin)
        done |= now
        y = new
    y = torch.where(done[..., None], fin, y)
    return _jacobian(th, y, chi_s, done.all(1)), y


def _exact_planes(d, slices, dev):
    """the multi-plane lens equation, one plane per slab of each replica"""
    chi_s, L = float(_chi(d["z_s"])), d["L"]
    pos, m = torch.as_tensor(d["pos"], device=dev), torch.as_tensor(d["mass"], device=dev) * MU_G
    rho, e2 = float(m.sum()) / L ** 3, float(d["soft"]) ** 2
    planes = []
    for j in range(len(d["rot"])):
        for s in range(slices):
            lo, hi = j * L + L / slices * s, min(j * L + L / slices * (s + 1), chi_s)
            if hi > lo:
                planes.append((j, s, lo, hi, 0.5 * (lo + hi)))
    th = _ray_angles(d, dev)
    slope, at = th.reshape(-1, 2).clone(), planes[0][4]
    x = at * slope

    def corner(u, v):
        return u * torch.atan(v / u) + 0.5 * v * torch.log(u * u + v * v)

    for q, (j, s, lo, hi, chi) in enumerate(planes):
        w = _placed(d, pos, j)
        on = (w[:, 2] < chi_s) & (torch.floor((w[:, 2] - j * L) / (L / slices)).clamp(max=slices - 1) == s)
        pj, mj = w[on, :2], m[on]
        defl = torch.zeros_like(x)
        chunk = max(1, (1 << 24) // x.shape[0])
        for a in range(0, pj.shape[0], chunk):
            dx, dy = (x[:, None, k] - pj[None, a:a + chunk, k] for k in range(2))
            f = mj[a:a + chunk] / (dx * dx + dy * dy + e2)
            defl[:, 0] += (f * dx).sum(1)
            defl[:, 1] += (f * dy).sum(1)
        u1, u0, v1, v0 = x[:, 0] + 0.5 * L, x[:, 0] - 0.5 * L, x[:, 1] + 0.5 * L, x[:, 1] - 0.5 * L
        defl[:, 0] -= rho * (hi - lo) * (corner(u1, v1) - corner(u0, v1) - corner(u1, v0) + corner(u0, v0))
        defl[:, 1] -= rho * (hi - lo) * (corner(v1, u1) - corner(v1, u0) - corner(v0, u1) + corner(v0, u0))
        slope = slope - 4.0 * (1.0 + float(_redshift(chi))) * defl
        x = x + ((planes[q + 1][4] if q + 1 < len(planes) else chi_s) - chi) * slope
    y = torch.zeros((*th.shape[:2], 8), dtype=torch.float64, device=dev)
    y[..., 1:3], y[..., 5:7], y[..., 3], y[..., 7] = x.view_as(th), slope.view_as(th), chi_s, 1.0
    return _jacobian(th, y, chi_s, torch.ones(th.shape[0], dtype=torch.bool, device=dev)), y


def _exact_born(d, dev):
    """convergence and shear from the Hessian of psi along the unperturbed rays"""
    chi_s, s, chi_l = float(_chi(d["z_s"])), d["asinh_s"], d["lens_chi"]
    x = _nodes(d["schedule"], d["steps"], chi_s, chi_l, s)
    du = (math.asinh((chi_s - chi_l) / s) - math.asinh(-chi_l / s)) / d["steps"]
    w = du * np.sqrt(s * s + (x - chi_l) ** 2) * x * (chi_s - x) / chi_s * (1.0 + _redshift(x))
    w[0] *= 0.5
    w[-1] *= 0.5
    th = torch.as_tensor(d["theta"], device=dev)
    pos, m = torch.as_tensor(d["pos"], device=dev), torch.as_tensor(d["mass"], device=dev) * MU_G
    e2 = torch.as_tensor(np.broadcast_to(np.asarray(d["soft"], np.float64) ** 2, d["mass"].shape).copy(), device=dev)
    out = torch.zeros((th.shape[0], 3), dtype=torch.float64, device=dev)
    chunk = max(1, (1 << 24) // th.shape[0])
    for xk, wk in zip(x.tolist(), w.tolist()):
        for a in range(0, pos.shape[0], chunk):
            q = pos[a:a + chunk]
            dx, dy = (th[:, None, k] * xk - q[None, :, k] for k in range(2))
            xx, yy = dx * dx, dy * dy
            i2 = 1.0 / (xx + yy + (xk - q[:, 2]) ** 2 + e2[a:a + chunk])
            m3 = m[a:a + chunk] * i2 * torch.sqrt(i2)
            m5 = m3 * i2
            out[:, 0] += wk * (2.0 * m3 - 3.0 * (xx + yy) * m5).sum(1)
            out[:, 1] += wk * 3.0 * ((yy - xx) * m5).sum(1)
            out[:, 2] -= wk * 6.0 * (dx * dy * m5).sum(1)
    return out
