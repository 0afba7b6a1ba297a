"""The work that users of the gridder have it do, as cases to be timed.

Every case is one call (or one short sequence of calls) of the public entry
points on inputs that are already on the GPU, with the plan (targets, kernel)
that a user's program keeps between calls.  Sizes are those of the workloads of
this repository (plain 2-D map, spectral cube, all-sky map, batch,
differentiable gridding, the paper's Example 1 and Appendix A.1) or generic.

``listed()`` names the cases, ``draw()`` gives further ones of the same
ranges, ``prepare()`` makes inputs and plan, ``run()`` is one pass, ``work()``
counts what a pass cannot do without, and ``exact()`` evaluates the same
result in 64 bits with plain torch.
"""
import math

import numpy as np
import torch

from paper_1604_06667_gb300 import Batch, Gridder, autograd

ARCMIN = 1.0 / 60.0
DEG = math.pi / 180.0
BATCH_CHANNELS = (1, 16, 64, 512)
BATCH_SIDES = (64, 128, 256, 512, 1024)


def _case(kind, **kw):
    """A case: samples ``n`` x channels ``c`` laid out as ``scan`` over a field
    of ``side`` degrees around (``lon0``, ``lat0``), ``nx`` x ``ny`` targets
    every ``pix`` arcmin, a kernel with parameters ``s1``, ``s2``, ``pa`` and
    support ``r`` (arcmin)."""
    c = dict(kind=kind, n=0, c=1, dtype="f32", scan="uniform", side=5.0, lon0=120.0, lat0=30.0,
             nx=100, ny=100, pix=3.0, kernel="gauss1d", s1=3.0, s2=0.0, pa=0.0, r=9.0,
             weighted=False, channel_major=False)
    c.update(kw)
    return c


def listed():
    return [
        # The smallest everyday call: one continuum map of 20,000 samples
        # (launches and host time count).
        _case("map", name="map_plain2d", n=20_000, side=5.0, lon0=30.0, lat0=0.0, pix=3.0,
              s1=2.5, r=7.5),
        # A spectral cube from a basket-weave raster: BF16 channels, the
        # tensor-core form.  The headline workload.
        _case("map", name="map_cube_bf16", n=1_000_000, c=256, dtype="bf16", scan="raster",
              side=10.0, nx=512, ny=512, pix=600.0 / 512, s1=3.0, r=9.0),
        # The same cube kept in FP32 throughout.
        _case("map", name="map_cube_f32", n=1_000_000, c=256, scan="raster", side=10.0, nx=512,
              ny=512, pix=600.0 / 512, s1=3.0, r=9.0),
        # A full-sky map of a few channels with an elliptical beam, poles and
        # longitude wrap included.
        _case("map", name="map_allsky_f32", n=10_000_000, c=32, scan="sky", nx=4096, ny=2048,
              kernel="gauss2d", s1=10.0, s2=6.0, pa=30.0, r=30.0),
        # The paper's Example 1 at its largest: 1e8 samples of one channel
        # onto 8,100 pixels.
        _case("map", name="map_example1", n=100_000_000, side=5.0, lon0=30.0, lat0=0.0, nx=90,
              ny=90, pix=200.0 / 60, s1=300.0 / 60 / math.sqrt(8 * math.log(2.0)),
              r=900.0 / 60 / math.sqrt(8 * math.log(2.0))),
        # Listing 1 of the paper from scratch on a new set of sight lines
        # (Appendix A.1: the pixel centres of a HEALPix grid): construct, set
        # the kernel, grid, normalise.
        _case("new_map", name="new_map_sightlines", n=11_796_480, scan="sky", nx=256, ny=0,
              s1=27.48 / math.sqrt(8 * math.log(2.0)), r=3 * 27.48 / math.sqrt(8 * math.log(2.0))),
        # Observing scans added one after the other with sample weights, an
        # odd channel count (a band after edge channels were cut), then the
        # cube and its weight map, channel-major as FITS stores it.
        _case("scans", name="scans_weighted_c37", n=200_000, c=37, scan="raster", side=5.0, nx=200,
              ny=200, pix=1.5, s1=3.0, r=9.0, weighted=True, channel_major=True),
        # Differentiable gridding: forward, adjoint and width gradient of one
        # training step (2e5 samples x 16 channels onto 256 x 256).
        _case("step", name="step_data_sigma", n=200_000, c=16, side=512.0 / 60, lon0=200.0,
              lat0=-20.0, nx=256, ny=256, pix=2.0, s1=4.0, r=12.0),
        # One iteration of continuum map making: the adjoint of the current
        # map, and the residual gridded on the same samples.
        _case("iterate", name="iterate_map_c1", n=1_000_000, c=1, side=512.0 / 60, lon0=200.0,
              lat0=-20.0, nx=512, ny=512, pix=1.0, s1=2.0, r=6.0),
        # A template cube interpolated at the positions of a scan.
        _case("interp", name="interp_c64", n=200_000, c=64, side=512.0 / 60, lon0=200.0,
              lat0=-20.0, nx=256, ny=256, pix=2.0, s1=4.0, r=12.0),
        # Channel flags: one weight (here 0 or 1) per sample and channel.
        _case("flags", name="flags_c128", n=250_000, c=128, scan="raster", side=5.0, nx=256, ny=256,
              pix=300.0 / 256, s1=3.0, r=9.0),
        # A batch of independent jobs of uneven size in one CUDA graph.
        _case("batch", name="batch_16", n=16, dtype="mixed", scan="uniform", lo=1e4, hi=1e6,
              fused=False, top_side=1024),
    ]


# ---------------------------------------------------------------------------
# Further cases of the same ranges
# ---------------------------------------------------------------------------
def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _int(rng, lo, hi):
    return int(round(_log(rng, lo, hi)))


def _field(rng, kind, n, c, nx, ny, s1, pix, **kw):
    """A plate-carree field of nx x ny pixels, moved off the poles."""
    side = max(nx, ny) * pix * ARCMIN
    lat0 = rng.uniform(-60.0, 60.0)
    lat0 = min(max(lat0, -85.0 + side / 2), 85.0 - side / 2)
    case = _case(kind, n=n, c=c, side=side, lon0=rng.uniform(0.0, 360.0), lat0=lat0, nx=nx, ny=ny,
                 pix=pix, s1=s1, r=3.0 * s1, scan=rng.choice(["uniform", "raster"]))
    case.update(kw)
    return case


def draw(rng):
    kind = rng.choice(["map", "map", "map", "map", "sky", "new_map", "scans", "step", "iterate",
                       "interp", "flags", "batch"])
    while True:
        case = _draw(rng, kind)
        w = work(case)
        pairs = _pairs(case) if kind != "batch" else 0.0
        # no more than the largest listed ones, and a field that the samples
        # cover where a fit or a kernel with negative lobes needs one
        if w["flops"] > 1.2e11 or w["bytes"] > 2.5e9 or pairs > 1.2e9:
            continue
        if kind in ("step", "iterate") and pairs * _channel_cost(case) > 1.5e9:
            continue
        if (kind == "step" or case["kernel"] == "tsinc") and pairs < 60.0 * _targets(case):
            continue
        return case


def _channel_cost(case):
    return 2.0 + case["c"] / 8.0


def _draw(rng, kind):
    s1 = _log(rng, 1.0, 8.0)
    pix = s1 * rng.uniform(0.35, 1.2)
    if kind == "map":
        nx = _int(rng, 48, 600)
        case = _field(rng, "map", _int(rng, 2e3, 3e6), rng.choice([1, 1, 3, 8, 16, 24, 37, 64, 100,
                                                                  128, 200, 256, 384, 512]),
                      nx, max(2, int(nx * rng.uniform(0.5, 1.0))), s1, pix,
                      dtype=rng.choice(["f32", "f32", "bf16"]), weighted=rng.random() < 0.3,
                      channel_major=rng.random() < 0.2)
        k = rng.random()
        if k < 0.2:
            case.update(kernel="gauss2d", s2=s1 * rng.uniform(0.4, 1.0), pa=rng.uniform(-90.0, 90.0))
        elif k < 0.3:
            # a tapered sin(x)/x with its first zeros inside the support
            case.update(kernel="tsinc", s1=0.8 * s1, s2=2.0 * s1)
        return case
    if kind == "sky":
        nx = 2 * _int(rng, 64, 1024)
        return _case("map", n=_int(rng, 1e5, 6e6), c=rng.choice([1, 4, 7, 16, 32]),
                     dtype=rng.choice(["f32", "bf16"]), scan="sky", nx=nx, ny=nx // 2,
                     kernel="gauss2d", s1=4.0 * s1 + 4.0, s2=3.0 * s1 + 3.0,
                     pa=rng.uniform(-90.0, 90.0), r=12.0 * s1 + 12.0)
    if kind == "new_map":
        ns = _int(rng, 16, 250)
        fw = 0.5 * 4.0 * math.degrees(math.sqrt(4.0 * math.pi / (12 * ns * ns))) / ARCMIN
        s1 = fw / math.sqrt(8 * math.log(2.0))
        return _case("new_map", n=int(12 * ns * ns * _log(rng, 4.0, 15.0)), c=rng.choice([1, 1, 2, 5]),
                     scan="sky", nx=ns, ny=0, s1=s1, r=3.0 * s1)
    if kind == "scans":
        nx = _int(rng, 64, 400)
        return _field(rng, "scans", _int(rng, 8e3, 6e5), rng.choice([1, 5, 16, 37, 75, 128, 201]), nx,
                      max(2, int(nx * rng.uniform(0.5, 1.0))), s1, pix, weighted=True,
                      channel_major=rng.random() < 0.5, dtype=rng.choice(["f32", "bf16"]))
    if kind == "step":
        nx = _int(rng, 48, 300)
        return _field(rng, "step", _int(rng, 2e4, 4e5), rng.choice([1, 3, 8, 16, 21, 32]), nx, nx,
                      s1, pix, scan="uniform")
    if kind == "iterate":
        nx = _int(rng, 64, 600)
        return _field(rng, "iterate", _int(rng, 2e4, 1e6), rng.choice([1, 1, 2, 8, 16]), nx, nx, s1,
                      pix)
    if kind == "interp":
        nx = _int(rng, 48, 400)
        case = _field(rng, "interp", _int(rng, 5e3, 4e5), rng.choice([1, 7, 16, 48, 64, 130]), nx, nx,
                      s1, pix)
        if rng.random() < 0.3:
            case.update(kernel="gauss2d", s2=s1 * rng.uniform(0.4, 1.0), pa=rng.uniform(-90.0, 90.0))
        return case
    if kind == "flags":
        nx = _int(rng, 48, 400)
        return _field(rng, "flags", _int(rng, 5e3, 4e5), rng.choice([1, 6, 16, 33, 64, 128]), nx, nx,
                      s1, pix, dtype=rng.choice(["f32", "bf16"]))
    hi = _log(rng, 1e5, 8e5)
    return _case("batch", n=rng.randint(3, 16), dtype=rng.choice(["mixed", "f32", "bf16"]), lo=1e4,
                 hi=hi, fused=rng.random() < 0.5, top_side=rng.choice([256, 512]))


# ---------------------------------------------------------------------------
# Sizes and work
# ---------------------------------------------------------------------------
def _targets(case):
    if case["kind"] == "new_map":
        return 12 * case["nx"] ** 2
    return case["nx"] * case["ny"]


def _pairs(case):
    """Expected (sample, target) pairs within the support."""
    r = case["r"] * ARCMIN
    if case["scan"] == "sky":
        area = 4.0 * math.pi / DEG ** 2
    else:
        area = case["side"] ** 2 * math.cos(case["lat0"] * DEG)
    return case["n"] * _targets(case) * math.pi * r * r / area


def _jobs(case):
    """The jobs of a batch: sizes that depend on the case alone."""
    rng = np.random.Generator(np.random.PCG64([case["n"], int(case["hi"]), case["top_side"]]))
    sides = [s for s in BATCH_SIDES if s <= case["top_side"]]
    jobs = []
    for j in range(case["n"]):
        n = int(round(10.0 ** rng.uniform(math.log10(case["lo"]), math.log10(case["hi"]))))
        c, side = int(rng.choice(BATCH_CHANNELS)), int(rng.choice(sides))
        if c == 512 and side == 1024:
            side = 512
        s1 = float(rng.uniform(1.0, 8.0))
        half = 0.25 * side * s1 * ARCMIN
        lat0 = float(np.clip(rng.uniform(-60.0, 60.0), -85.0 + min(half, 80.0), 85.0 - min(half, 80.0)))
        dtype = case["dtype"] if case["dtype"] != "mixed" else ("bf16" if j % 2 else "f32")
        jobs.append(_case("map", n=n, c=c, dtype=dtype, side=2.0 * half,
                          lon0=float(rng.uniform(0.0, 360.0)), lat0=lat0, nx=side, ny=side,
                          pix=0.5 * s1, s1=s1, r=3.0 * s1))
    return jobs


def work(case):
    """Each input and output once; two operations per pair and channel."""
    if case["kind"] == "batch":
        parts = [work(j) for j in _jobs(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    n, c, P = case["n"], case["c"], _targets(case)
    width = 2 if case["dtype"] == "bf16" else 4
    flops = 2.0 * c * _pairs(case)
    coords, data, out = 16.0 * n, width * n * c, 4.0 * P * c
    kind = case["kind"]
    if kind in ("map", "new_map", "scans"):
        b = coords + data + out + (4.0 * n if case["weighted"] else 0.0)
        if kind == "new_map":
            b += 16.0 * P
        if kind == "scans":
            b += 4.0 * P
        return {"bytes": b, "flops": flops}
    if kind == "step":        # data and coordinates in, map and data gradient out, target map in
        return {"bytes": coords + 2.0 * data + 2.0 * out, "flops": 3.0 * flops}
    if kind == "iterate":     # map and data in, residual out, gradient map out
        return {"bytes": 2.0 * data + 2.0 * out, "flops": 2.0 * flops}
    if kind == "interp":      # map in, samples out
        return {"bytes": out + data, "flops": flops}
    return {"bytes": coords + data + 4.0 * n * c + 2.0 * out, "flops": 2.0 * flops}   # flags


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _rand(g, n, dtype=torch.float64):
    return torch.rand(n, generator=g, device="cuda", dtype=dtype)


def _samples(case, g):
    """Sample coordinates in degrees."""
    n, side = case["n"], case["side"]
    if case["scan"] == "sky":
        lat = torch.rad2deg(torch.asin(2.0 * _rand(g, n) - 1.0))
        return 360.0 * _rand(g, n), lat
    if case["scan"] == "uniform":
        return case["lon0"] + (_rand(g, n) - 0.5) * side, case["lat0"] + (_rand(g, n) - 0.5) * side
    # basket weave: zig-zag scans along longitude, then along latitude, twice
    # as dense along a scan as across, with pointing jitter
    rows = max(1, int(math.sqrt(n / 3.3)))
    along = 2 * rows
    k = torch.arange(n, device="cuda")
    first = k < rows * along
    q = torch.where(first, k, k - rows * along)
    row = q // along
    step = q % along
    step = torch.where(row % 2 == 1, along - 1 - step, step)
    a = (row.double() % rows + 0.5) / rows - 0.5
    b = (step.double() + 0.5) / along - 0.5
    jit = 0.2 * side / rows
    dl = torch.where(first, b, a) * side + jit * torch.randn(n, generator=g, device="cuda", dtype=torch.float64)
    db = torch.where(first, a, b) * side + jit * torch.randn(n, generator=g, device="cuda", dtype=torch.float64)
    return case["lon0"] + dl, case["lat0"] + db


def _scene(case, seed, count=6):
    """A few smooth sources: directions, width, amplitudes, line profiles."""
    g = _gen(seed + 1_000_003)
    if case["scan"] == "sky":
        lat = torch.rad2deg(torch.asin(2.0 * _rand(g, count) - 1.0))
        lon, sig = 360.0 * _rand(g, count), 4.0
    else:
        lon = case["lon0"] + (_rand(g, count) - 0.5) * case["side"]
        lat = case["lat0"] + (_rand(g, count) - 0.5) * case["side"]
        sig = 4.0 * case["s1"] * ARCMIN
    c = case["c"]
    amp = 1.0 + 9.0 * _rand(g, count).float()
    k = torch.arange(c, device="cuda", dtype=torch.float32)
    c0 = _rand(g, count).float() * c
    prof = torch.exp(-0.5 * ((k[None, :] - c0[:, None]) / (0.1 * c + 1.0)) ** 2)
    return _unit(lon, lat), sig * DEG, amp[:, None] * prof


def _add_sky(data, scene, lon, lat):
    """The sources' values at given directions added to ``data`` [n, c]."""
    v, sig, prof = scene
    for a in range(0, lon.numel(), 1 << 22):
        u = _unit(lon[a:a + (1 << 22)], lat[a:a + (1 << 22)])
        data[a:a + (1 << 22)] += torch.exp((u @ v.T - 1.0) / (sig * sig)).float() @ prof
    return data


def _values(case, lon, lat, seed, g):
    """Channel values: smooth sources with a line profile each, plus noise."""
    data = torch.randn((lon.numel(), case["c"]), generator=g, device="cuda", dtype=torch.float32)
    if case["scan"] == "sky":
        data *= 0.1
    _add_sky(data, _scene(case, seed), lon, lat)
    return data.to(torch.bfloat16) if case["dtype"] == "bf16" else data


def _target_grid(case):
    """Target coordinates in degrees: a plate-carree field, the whole sky, or
    the pixel centres of a HEALPix grid."""
    nx, ny = case["nx"], case["ny"]
    if case["kind"] == "new_map":
        return _healpix_centres(nx)
    if case["scan"] == "sky":
        xs = (torch.arange(nx, device="cuda", dtype=torch.float64) + 0.5) * (360.0 / nx)
        ys = -90.0 + (torch.arange(ny, device="cuda", dtype=torch.float64) + 0.5) * (180.0 / ny)
    else:
        d = case["pix"] * ARCMIN
        xs = case["lon0"] + (torch.arange(nx, device="cuda", dtype=torch.float64) - 0.5 * (nx - 1)) * d
        ys = case["lat0"] + (torch.arange(ny, device="cuda", dtype=torch.float64) - 0.5 * (ny - 1)) * d
    lat, lon = torch.meshgrid(ys, xs, indexing="ij")
    return lon.reshape(-1).contiguous(), lat.reshape(-1).contiguous()


def _healpix_centres(ns):
    """RING-scheme pixel centres (Gorski et al. 2005)."""
    i = np.arange(1, 4 * ns)
    cap = np.minimum(i, 4 * ns - i)
    m = np.where(cap < ns, 4 * cap, 4 * ns)
    z = np.where(cap < ns, 1.0 - cap * cap / (3.0 * ns * ns), 4.0 / 3.0 - 2.0 * i / (3.0 * ns))
    z = np.where((cap < ns) & (i > 2 * ns), -z, z)
    shift = np.where(cap < ns, 0.5, 0.5 * ((i - ns + 1) % 2))
    m, shift, lat = (torch.from_numpy(v).cuda() for v in (m, shift, np.degrees(np.arcsin(z))))
    start = torch.cumsum(m, 0) - m
    ring = torch.repeat_interleave(torch.arange(m.numel(), device="cuda"), m)
    j = torch.arange(ring.numel(), device="cuda") - start[ring]
    return (j + shift[ring]) * (360.0 / m[ring]), lat[ring].contiguous()


def _kernel(case):
    """Arguments of set_kernel: type, parameters, support, index resolution."""
    s1, s2 = case["s1"] * ARCMIN, case["s2"] * ARCMIN
    if case["kernel"] == "gauss2d":
        return "gauss2d", (s1, s2, case["pa"]), case["r"] * ARCMIN, 0.5 * min(s1, s2)
    if case["kernel"] == "tsinc":
        return "tsinc", (s1, s2), case["r"] * ARCMIN, 0.25 * s2
    return "gauss1d", (s1,), case["r"] * ARCMIN, 0.5 * s1


def _gridder(case):
    lon_t, lat_t = _target_grid(case)
    g = Gridder(lon_t, lat_t, n_channels=case["c"])
    g.set_kernel(*_kernel(case))
    return g


def _inputs(case, seed):
    g = _gen(seed)
    lon, lat = _samples(case, g)
    data = _values(case, lon, lat, seed, g)
    om = 0.25 + _rand(g, lon.numel()).float() if case["weighted"] else None
    return lon, lat, data, om, g


def _scan_parts(case):
    """Eight scans of uneven length (the first sample of each, and the end)."""
    n = case["n"]
    return [int(n * f) for f in (0.0, 0.07, 0.21, 0.33, 0.5, 0.61, 0.79, 0.9, 1.0)]


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind == "batch":
        jobs, keep = [], []
        for k, job in enumerate(_jobs(case)):
            lon, lat, data, _, _ = _inputs(job, seed * 64 + k)
            g = _gridder(job)
            out = torch.empty((g.n_targets, g.n_channels), device="cuda")
            jobs.append((g, lon, lat, data, out))
            keep.append(out)
        st["batch"] = Batch(jobs, n_streams=16).set_fused(case["fused"]).capture()
        st["out"] = keep
        return st
    lon, lat, data, om, g = _inputs(case, seed)
    st.update(lon=lon, lat=lat, data=data, om=om)
    if kind == "new_map":
        st["lon_t"], st["lat_t"] = _target_grid(case)
        return st
    gr = st["gridder"] = _gridder(case)
    if kind == "scans":
        p = _scan_parts(case)
        st["parts"] = [(lon[a:b], lat[a:b], data[a:b], om[a:b]) for a, b in zip(p, p[1:])]
    elif kind == "step":
        # the fit's target: the sources at the pixels, without noise
        st["goal"] = _goal(case, seed)
        st["data"] = data.requires_grad_()
        st["sigma"] = torch.tensor(case["s1"] * ARCMIN, device="cuda", requires_grad=True)
    elif kind == "iterate":
        st["W"] = torch.empty(gr.n_targets, device="cuda")
        st["map"] = gr.grid_oneshot(lon, lat, data, out_weights=st["W"]).nan_to_num_()
    elif kind == "interp":
        gr.grid_oneshot(lon, lat, data)          # the positions to interpolate at
        st["map"] = _goal(case, seed)
    elif kind == "flags":
        st["flags"] = (_rand(g, lon.numel() * case["c"], torch.float32) > 0.1).float().reshape(-1, case["c"])
    return st


def _goal(case, seed):
    """The noiseless sources at the target positions, [P, C]."""
    lon_t, lat_t = _target_grid(case)
    return _add_sky(torch.zeros((lon_t.numel(), case["c"]), device="cuda"), _scene(case, seed), lon_t,
                    lat_t)


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "batch":
        st["batch"].run()
        return st["out"]
    if kind == "new_map":
        g = Gridder(st["lon_t"], st["lat_t"], n_channels=case["c"])
        g.set_kernel(*_kernel(case))
        g.grid(st["lon"], st["lat"], st["data"])
        return g.get_datacube()
    g = st["gridder"]
    if kind == "map":
        return g.grid_oneshot(st["lon"], st["lat"], st["data"], weights=st["om"],
                              channel_major=case["channel_major"])
    if kind == "scans":
        g.reset()
        for lon, lat, data, om in st["parts"]:
            g.grid(lon, lat, data, weights=om)
        w = torch.empty(g.n_targets, device="cuda")
        return g.get_datacube(channel_major=case["channel_major"], out_weights=w), w
    if kind == "step":
        _, _, r, maxres = _kernel(case)
        R = autograd.grid(g, st["lon"], st["lat"], st["data"], st["sigma"], r, maxres)
        loss = 0.5 * (R - st["goal"]).square().sum()
        gd, gs = torch.autograd.grad(loss, (st["data"], st["sigma"]))
        return R.detach(), gd, gs
    if kind == "iterate":
        res = g.degrid(st["map"], map_weights=st["W"]) - st["data"]
        return res, g.grid_oneshot(None, None, res)
    if kind == "interp":
        w = torch.empty(case["n"], device="cuda")
        return g.interp(st["map"], out_weights=w), w
    w = torch.empty((g.n_targets, case["c"]), device="cuda")
    return g.grid_oneshot_pcw(st["lon"], st["lat"], st["data"], st["flags"], out_weights=w), w


# ---------------------------------------------------------------------------
# The same in 64 bits with plain torch
# ---------------------------------------------------------------------------
def _unit(lon, lat):
    l, b = lon.double() * DEG, lat.double() * DEG
    return torch.stack([torch.cos(b) * torch.cos(l), torch.cos(b) * torch.sin(l), torch.sin(b)], -1)


def _leaves(u, size):
    """Indices of u's rows in compact groups of ``size`` (the last ones are
    padded by repeating -1), by halving along the widest axis."""
    n = u.shape[0]
    k = 1
    while k * size < n:
        k *= 2
    idx = torch.full((k * size,), -1, device=u.device, dtype=torch.int64)
    idx[:n] = torch.arange(n, device=u.device)
    idx = idx[None, :]
    while idx.shape[1] > size:
        v = u[idx.clamp_min(0)]
        lo = torch.where(idx[..., None] < 0, math.inf, v).amin(1)
        hi = torch.where(idx[..., None] < 0, -math.inf, v).amax(1)
        axis = (hi - lo).argmax(1)
        key = torch.gather(v, 2, axis[:, None, None].expand(-1, idx.shape[1], 1))[..., 0]
        key = torch.where(idx < 0, math.inf, key)
        idx = torch.gather(idx, 1, key.argsort(1)).reshape(2 * idx.shape[0], -1)
    return idx


def _reach(c, rad, u, idx, r):
    """The entries of ``idx`` within rad + r (chords) of the centre c."""
    d = u[idx] - c
    return idx[(d * d).sum(1) <= (rad + r) ** 2]


def _pair_blocks(ut, us, chord, limit=1 << 25):
    """(targets, samples) index blocks that hold every pair within ``chord``."""
    size = 128 if ut.shape[0] <= 1 << 20 else 512
    leaf = _leaves(ut, size)
    group = max(1, min(64, leaf.shape[0]))
    every = torch.arange(us.shape[0], device=us.device)
    for a in range(0, leaf.shape[0], group):
        part = leaf[a:a + group]
        if bool((part < 0).all()):
            continue
        v = ut[part[part >= 0]]
        c = v.mean(0)
        rad = float((v - c).norm(dim=1).max())
        near = _reach(c, rad, us, every, chord) if leaf.shape[0] > group else every
        for row in part:
            ti = row[row >= 0]
            if not ti.numel():
                continue
            c = ut[ti].mean(0)
            rad = float((ut[ti] - c).norm(dim=1).max())
            si = _reach(c, rad, us, near, chord * (1 + 1e-9))
            step = max(1, limit // ti.numel())
            for b in range(0, si.numel(), step):
                yield ti, si[b:b + step]


class _Exact:
    def __init__(self, case, lon, lat):
        self.case = case
        lon_t, lat_t = _target_grid(case)
        self.ut, self.us = _unit(lon_t, lat_t), _unit(lon, lat)
        self.P, self.N = lon_t.numel(), lon.numel()
        _, p, r, _ = _kernel(case)
        self.chord = 2.0 * math.sin(0.5 * r * DEG)
        self.p = [v * DEG for v in p]
        if case["kernel"] == "gauss2d":
            l, b, pa = lon_t * DEG, lat_t * DEG, self.p[2]
            e = torch.stack([-torch.sin(l), torch.cos(l), torch.zeros_like(l)], -1)
            n = torch.stack([-torch.sin(b) * torch.cos(l), -torch.sin(b) * torch.sin(l), torch.cos(b)], -1)
            self.f1 = n * math.cos(pa) + e * math.sin(pa)
            self.f2 = e * math.cos(pa) - n * math.sin(pa)

    def blocks(self):
        """(ti, si, w, d) of every block, w = 0 outside the support."""
        kernel, p = self.case["kernel"], self.p
        for ti, si in _pair_blocks(self.ut, self.us, self.chord):
            t, s = self.ut[ti], self.us[si]
            dx = [t[:, k, None] - s[None, :, k] for k in range(3)]
            c2 = dx[0] * dx[0] + dx[1] * dx[1] + dx[2] * dx[2]
            d = 2.0 * torch.asin((0.5 * c2.sqrt()).clamp_max(1.0))
            if kernel == "gauss2d":
                ap, bp = (sum(dx[k] * f[ti][:, k, None] for k in range(3)) for f in (self.f1, self.f2))
                s2 = ap * ap + bp * bp
                q = torch.where(s2 > 0, d * d / s2, 1.0)
                w = torch.exp(-0.5 * q * ((ap / p[0]) ** 2 + (bp / p[1]) ** 2))
            elif kernel == "tsinc":
                w = torch.sinc(d / p[0]) * torch.exp(-(d / p[1]) ** 2)
            else:
                w = torch.exp(-0.5 * (d / p[0]) ** 2)
            yield ti, si, torch.where(c2 <= self.chord ** 2, w, 0.0), d

    def grid(self, data, om=None):
        """Numerator [P, C] and weight map [P]."""
        num = torch.zeros((self.P, data.shape[1]), device="cuda", dtype=torch.float64)
        W = torch.zeros(self.P, device="cuda", dtype=torch.float64)
        for ti, si, w, _ in self.blocks():
            if om is not None:
                w = w * om[si].double()
            num[ti] += w @ data[si].double()
            W[ti] += w.sum(1)
        return num, W


def _ratio(num, W):
    return torch.where(W > 0, num / W, math.nan)


def _exact_map(case, lon, lat, data, om):
    num, W = _Exact(case, lon, lat).grid(data, om)
    return _ratio(num, W[:, None]), W


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        outs = []
        for k, job in enumerate(_jobs(case)):
            lon, lat, data, _, _ = _inputs(job, seed * 64 + k)
            outs.append(_exact_map(job, lon, lat, data, None)[0])
        return outs
    lon, lat, data, om, g = _inputs(case, seed)
    if kind in ("map", "new_map"):
        R = _exact_map(case, lon, lat, data, om)[0]
        return R.T.contiguous() if case["channel_major"] else R
    if kind == "scans":
        R, W = _exact_map(case, lon, lat, data, om)
        return (R.T.contiguous() if case["channel_major"] else R), W
    ex = _Exact(case, lon, lat)
    if kind == "flags":
        fl = (_rand(g, lon.numel() * case["c"], torch.float32) > 0.1).float().reshape(-1, case["c"])
        both, _ = ex.grid(torch.cat([fl * data.float(), fl], 1))
        num, W = both[:, :case["c"]], both[:, case["c"]:]
        return _ratio(num, W), W
    if kind == "interp":
        y = _goal(case, seed).double()
        x = torch.zeros((ex.N, y.shape[1]), device="cuda", dtype=torch.float64)
        v = torch.zeros(ex.N, device="cuda", dtype=torch.float64)
        for ti, si, w, _ in ex.blocks():
            x.index_add_(0, si, w.T @ y[ti])
            v.index_add_(0, si, w.sum(0))
        return _ratio(x, v[:, None]), v
    num, W = ex.grid(data)
    R, Wi = _ratio(num, W[:, None]), torch.where(W > 0, 1.0 / W, 0.0)
    x = torch.zeros((ex.N, case["c"]), device="cuda", dtype=torch.float64)
    if kind == "iterate":
        m = R.float().nan_to_num_().double() * Wi[:, None]
        for ti, si, w, _ in ex.blocks():
            x.index_add_(0, si, w.T @ m[ti])
        x -= data.double()
        num, W = ex.grid(x)
        return x, _ratio(num, W[:, None])
    # step: residual, its adjoint, and its product with dR/dsigma
    res = R - _goal(case, seed).double()
    s = case["s1"] * ARCMIN
    n1, w1 = torch.zeros_like(num), torch.zeros_like(W)
    for ti, si, w, d in ex.blocks():
        x.index_add_(0, si, w.T @ (res[ti] * Wi[ti, None]))
        w = w * (d / DEG) ** 2 / s ** 3
        n1[ti] += w @ data[si].double()
        w1[ti] += w.sum(1)
    gs = (res * (n1 - R * w1[:, None]) * Wi[:, None]).sum()
    return R, x, gs
