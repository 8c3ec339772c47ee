"""What this framework is timed on: the calls that its users make, over the range of sizes they make them at.

A case is a dict of plain values; ``prepare`` makes its inputs from a seed (coronae, views, weights), ``run`` is one
pass through the public Python API, ``exact`` the same method in 64 bits as plain torch gives it.  The sizes are those
of this repository's workloads and tests, or cuts of them that take under two seconds.

    kind      the call
    map       Context.trace_image on a loaded corona
    batch     BatchPlan.launch: many small requests as one plan
    spectrum  trace_image without magnification, then disk_mean_tb: the disk-mean spectrum
    snapshot  load_grid from pinned host memory, then trace_image: one frame of a sequence of coronae
    tape      trace_image_tape and Tape.backward: a map and the gradient of its misfit
    autograd  RayTraceFn forward and backward: one step of a fit, the corona a tensor
    beam      beam_convolve of finished maps
    disk      disk_mean_tb of finished maps
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2606_02413_gb300 as rt

DEV = "cuda"


# --------------------------------------------------------------------------------------------------------- the cases

def _map(name, **kw):
    c = {"name": name, "kind": "map", "corona": "log", "n_r": 64, "n_t": 32, "n_p": 64, "r_max": 4.0, "f64": False,
         "nx": 64, "ny": 64, "extent": 2.5, "lon": 0.0, "lat": 0.0, "nf": 1, "f_lo": 100e6, "f_hi": 100e6,
         "dtau": 2e-3, "mode": rt.RT_STEPWISE, "nb": 4, "mixed": True}
    c.update(kw)
    return c


def listed():
    return [
        # The smallest useful call: one 64^2 map at one frequency (a quick look, or one iteration of an interactive
        # view).  4096 rays do not fill the GPU: what counts is how long one ray's steps take.
        _map("map-64x64-1f", f64=True),
        # An odd image from an oblique observer on an odd grid, in the default plain form with 8 neighbours.
        _map("map-97x61-3f-8nb-plain", n_r=65, n_t=33, n_p=63, nx=97, ny=61, lon=1.1, lat=0.35, nf=3, f_lo=60e6,
             f_hi=300e6, nb=8, mixed=False),
        # The main workload (a global corona out to 30 R_sun, 16 maps over 40-800 MHz, 4 neighbours, compensated
        # form), its 512^2 image cut to 128^2.  The largest case.
        _map("global-128x128-16f", corona="global", n_r=256, n_t=180, n_p=360, r_max=30.0, nx=128, ny=128,
             extent=3.0, nf=16, f_lo=40e6, f_hi=800e6),
        # The fine grid of the precision workload (512x360x720, 8 neighbours), 1024^2 x 32 cut to 96^2 x 4: cells
        # hardly wider than the neighbours' offsets.
        _map("fine-96x96-4f-8nb", n_r=512, n_t=360, n_p=720, nx=96, ny=96, nf=4, f_lo=40e6, f_hi=800e6, nb=8),
        # Persistent neighbours (tube mode), the step-converged magnification.
        _map("tube-96x96-2f", nx=96, ny=96, nf=2, f_lo=150e6, f_hi=400e6, mode=rt.RT_TUBE),
        # A service's batch: 40 small requests (sides 16-64, 1-4 frequencies, any longitude) as one planned launch.
        _map("batch-40", kind="batch", n_req=40, side_lo=16, side_hi=64, nf=4, f_lo=40e6, f_hi=800e6),
        # The disk-mean spectrum without the magnification term: 8 maps traced, each reduced to its mean.
        _map("spectrum-128x128-8f", kind="spectrum", nx=128, ny=128, nf=8, f_lo=40e6, f_hi=400e6,
             mode=rt.RT_MAG_OFF, mixed=False),
        # One frame of a sequence of coronae: the 256x180x360 grid comes from the host, two maps are traced.
        _map("snapshot-96x96-2f", kind="snapshot", corona="global", n_r=256, n_t=180, n_p=360, r_max=30.0, nx=96,
             ny=96, extent=3.0, nf=2, f_lo=80e6, f_hi=300e6),
        # The differentiation workload's corona, 256^2 x 8 cut to 128^2 x 8: forward with its tape, reverse sweep.
        _map("tape-128x128-8f", kind="tape", n_r=128, n_t=90, n_p=180, nx=128, ny=128, nf=8, f_lo=40e6, f_hi=400e6),
        # One step of a fit through autograd on a small corona: the grid is loaded, traced and differentiated.
        _map("autograd-40x40-2f", kind="autograd", n_r=96, n_t=64, n_p=128, nx=40, ny=40, nf=2, f_lo=80e6,
             f_hi=300e6),
        # The comparison products of the 512^2 x 16 maps: beam-convolved maps, and the disk-mean spectrum.
        {"name": "beam-512x512-16f", "kind": "beam", "nx": 512, "ny": 512, "extent": 3.0, "nf": 16, "f_lo": 40e6,
         "f_hi": 800e6, "baseline": 15e3},
        {"name": "disk-512x512-16f", "kind": "disk", "nx": 512, "ny": 512, "extent": 3.0, "nf": 16, "f_lo": 40e6,
         "f_hi": 800e6, "radius": 0.5},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _band(rng, nf):
    lo = _log(rng, 40e6, 400e6)
    return {"nf": nf, "f_lo": lo, "f_hi": lo if nf == 1 else lo * rng.uniform(1.5, min(10.0, 800e6 / lo))}


def _image(rng, lo, hi):
    return {"nx": int(round(_log(rng, lo, hi))), "ny": int(round(_log(rng, lo, hi))),
            "lon": rng.uniform(0.0, 6.28), "lat": rng.uniform(-0.6, 0.6)}


def draw(rng):
    kind = rng.choice(["map", "map", "map", "global", "batch", "spectrum", "tape", "autograd", "beam", "disk"])
    if kind in ("beam", "disk"):
        c = {"kind": kind, "nx": rng.randint(40, 640), "ny": rng.randint(40, 640), "extent": 3.0}
        c.update(_band(rng, rng.randint(1, 16)))
        if kind == "beam":
            c["baseline"] = rng.uniform(5e3, 15e3)
        else:
            c["radius"] = rng.uniform(0.3, 1.5)
        return c
    c = _map("", kind=kind, n_r=rng.randint(40, 160), n_t=rng.randint(24, 96), n_p=rng.randint(40, 192))
    del c["name"]
    c["dtau"] = rng.choice([1e-3, 2e-3, 4e-3])
    c["mixed"] = rng.random() < 0.6
    if kind == "global":
        c.update(kind="map", corona="global", n_r=256, n_t=180, n_p=360, r_max=30.0, extent=3.0, dtau=2e-3)
        c.update(_image(rng, 20, 110))
        c.update(_band(rng, rng.randint(1, 8)))
    elif kind == "map":
        c.update(_image(rng, 17, 200))
        c.update(_band(rng, rng.randint(1, 8)))
        c["nb"] = rng.choice([2, 4, 4, 8])
        c["f64"] = rng.random() < 0.3
    elif kind == "batch":
        c.update(_band(rng, rng.randint(1, 4)))
        c.update(n_req=rng.randint(4, 56), side_lo=16, side_hi=rng.randint(24, 72))
    elif kind == "spectrum":
        c.update(_image(rng, 30, 200), mode=rt.RT_MAG_OFF)
        c.update(_band(rng, rng.randint(2, 12)))
    elif kind == "tape":
        c.update(_image(rng, 24, 100))
        c.update(_band(rng, rng.randint(1, 8)))
        c["mode"] = rng.choice([rt.RT_STEPWISE, rt.RT_STEPWISE, rt.RT_MAG_OFF])
    else:
        c.update(_image(rng, 16, 64))
        c.update(_band(rng, rng.randint(1, 4)))
    return c


# -------------------------------------------------------------------------------------------------------- the inputs

class View:
    def __init__(self, lon, lat, nx, ny, extent):
        # square pixels: the shorter side spans less
        ex, ey = extent * nx / max(nx, ny), extent * ny / max(nx, ny)
        self.lon_rad, self.lat_rad, self.nx, self.ny = lon, lat, nx, ny
        self.x0, self.x1, self.y0, self.y1 = -ex, ex, -ey, ey


def _view(c):
    return View(c.get("lon", 0.0), c.get("lat", 0.0), c["nx"], c["ny"], c["extent"])


def _freqs(c):
    if c["nf"] == 1:
        return np.array([c["f_lo"]])
    return c["f_lo"] * (c["f_hi"] / c["f_lo"]) ** (np.arange(c["nf"]) / (c["nf"] - 1.0))


def _corona(c, seed):
    """(r, theta, phi, n_e, T_e): Newkirk background on a log grid with smooth seeded structure, or the global corona
    (stretched grid, lognormal modulation of 0.1 R_sun, active regions, polar holes)."""
    rng = np.random.Generator(np.random.PCG64(seed))
    n_r, n_t, n_p = c["n_r"], c["n_t"], c["n_p"]
    i = np.arange(n_r, dtype=np.float64) / (n_r - 1)
    if c["corona"] == "global":
        r = 1.0 + (c["r_max"] - 1.0) * np.expm1(5.0 * i) / math.expm1(5.0)
    else:
        r = c["r_max"] ** i
    th = (np.arange(n_t) + 0.5) * math.pi / n_t
    ph = np.arange(n_p) * (2.0 * math.pi / n_p)
    R = torch.tensor(r, device=DEV)[:, None, None]
    T = torch.tensor(th, device=DEV)[None, :, None]
    P = torch.tensor(ph, device=DEV)[None, None, :]
    base = 4.2e4 * 10.0 ** (4.32 / R)
    if c["corona"] != "global":
        # a few smooth modes in (r, theta, phi); T_e around 1 MK
        g = torch.zeros((), dtype=torch.float64, device=DEV)
        t = torch.zeros((), dtype=torch.float64, device=DEV)
        for _ in range(4):
            m = int(rng.integers(1, 4))
            a, b, s, q = rng.normal(), rng.uniform(0, 6.28), rng.uniform(0, 6.28), rng.uniform(1.0, 3.0)
            mode = torch.sin(T) ** m * torch.cos(m * P + b) * torch.cos(q * torch.log(R) + s)
            g = g + a * mode
            t = t + rng.normal() * mode
        ne = base * torch.exp(0.12 * g)
        te = 1.0e6 * torch.exp(0.08 * t)
        dt = torch.float64 if c["f64"] else torch.float32
        return r, th, ph, ne.to(dt).contiguous(), te.to(dt).contiguous()
    Rf, Tf, Pf = R.float(), T.float(), P.float()
    x, y, z = Rf * (torch.sin(Tf) * torch.cos(Pf)), Rf * (torch.sin(Tf) * torch.sin(Pf)), Rf * torch.cos(Tf)
    z = z.expand_as(x)
    n_modes, corr = 256, 0.1
    k = torch.tensor(rng.normal(0.0, 1.0 / corr, size=(3, n_modes)), dtype=torch.float32, device=DEV)
    s = torch.tensor(rng.uniform(0.0, 2.0 * math.pi, size=n_modes), dtype=torch.float32, device=DEV)
    pts = torch.stack([x.reshape(-1), y.reshape(-1), z.reshape(-1)], 1)
    g = torch.empty(pts.shape[0], device=DEV)
    for b in range(0, pts.shape[0], 1 << 20):
        g[b:b + (1 << 20)] = torch.cos(pts[b:b + (1 << 20)] @ k + s).sum(1)
    g = g.reshape(x.shape) * math.sqrt(2.0 / n_modes)
    ne = base.float() * torch.exp(0.3 * g - 0.045)
    te = torch.full_like(ne, 1.0e6)
    for _ in range(6):
        u, lon = rng.uniform(-1.0, 1.0), rng.uniform(0.0, 2.0 * math.pi)
        s0 = math.sqrt(1.0 - u * u)
        cx, cy, cz = 1.05 * s0 * math.cos(lon), 1.05 * s0 * math.sin(lon), 1.05 * u
        amp, tb, rad = rng.uniform(5.0, 20.0), rng.uniform(2.0e6, 3.0e6), rng.uniform(0.05, 0.15)
        blob = torch.exp(-((x - cx) ** 2 + (y - cy) ** 2 + (z - cz) ** 2) / (2.0 * rad * rad))
        ne *= 1.0 + (amp - 1.0) * blob
        te += (tb - te) * blob
    edge = math.radians(3.0)
    hole = 0.5 * (1 + torch.tanh((math.radians(30) - Tf) / edge)) + 0.5 * (1 + torch.tanh((Tf - math.radians(150)) / edge))
    ne *= 1.0 - 0.7 * hole.clamp(max=1.0)
    return r, th, ph, ne.contiguous(), te.contiguous()


def _maps(c, seed):
    """Finished T_b maps [nf, ny, nx]: a 1 MK disk with limb and small-scale structure."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    v = _view(c)
    u = v.x0 + (torch.arange(v.nx, device=DEV) + 0.5) * (v.x1 - v.x0) / v.nx
    w = v.y0 + (torch.arange(v.ny, device=DEV) + 0.5) * (v.y1 - v.y0) / v.ny
    b = torch.sqrt(u[None, None, :] ** 2 + w[None, :, None] ** 2)
    rad = 1.0 + 0.5 * torch.rand((c["nf"], 1, 1), generator=gen, device=DEV)
    n = torch.randn((c["nf"], v.ny, v.nx), generator=gen, device=DEV)
    return (1.0e6 / (1.0 + torch.exp((b - rad) / 0.08)) * (1.0 + 0.05 * n)).float().contiguous()


def _weights(c, seed):
    """dL/dT_b of a misfit: residuals of about a tenth of the maps."""
    gen = torch.Generator(device=DEV).manual_seed(seed + 1)
    return (2.0e5 * torch.randn((c["nf"], c["ny"], c["nx"]), generator=gen, device=DEV)).contiguous()


def _requests(c, seed):
    """The batch's requests: sides and frequency counts from the case, longitudes and frequencies from the seed."""
    shape = np.random.Generator(np.random.PCG64([c["n_req"], c["side_lo"], c["side_hi"], c["nf"]]))
    rng = np.random.Generator(np.random.PCG64(seed + 2))
    out = []
    for _ in range(c["n_req"]):
        side = int(shape.integers(c["side_lo"], c["side_hi"] + 1))
        nf = int(shape.integers(1, c["nf"] + 1))
        f = np.exp(rng.uniform(math.log(c["f_lo"]), math.log(c["f_hi"] * 1.0001), size=nf))
        out.append((View(float(rng.uniform(0.0, 2.0 * math.pi)), 0.0, side, side, c["extent"]), f))
    return out


def _options(c):
    return rt.options(dtau=c["dtau"], s_mode=c["mode"], n_nb=c["nb"],
                      precision=rt.RT_MIXED if c["mixed"] else rt.RT_PLAIN_F32)


class _Request:
    def __init__(self, view, freqs_hz):
        self.view, self.freqs_hz = view, freqs_hz


def prepare(case, seed):
    c, kind = case, case["kind"]
    s = {"case": c, "ctx": rt.Context(0)}
    if kind in ("beam", "disk"):
        s.update(view=_view(c), freqs=_freqs(c), tb=_maps(c, seed))
        return s
    r, th, ph, ne, te = _corona(c, seed)
    s.update(axes=(r, th, ph), view=_view(c), freqs=_freqs(c), opts=_options(c))
    if kind == "snapshot":
        s.update(ne=ne.cpu().pin_memory().numpy(), te=te.cpu().pin_memory().numpy())
        return s
    if kind == "autograd":
        s.update(ne=ne.requires_grad_(True), te=te.requires_grad_(True), w=_weights(c, seed))
        return s
    s["grid"] = s["ctx"].load_grid(r, th, ph, ne, te)
    if kind == "batch":
        s["plan"] = s["ctx"].batch_plan(s["grid"], [_Request(v, f) for v, f in _requests(c, seed)], s["opts"])
    if kind == "tape":
        s["w"] = _weights(c, seed)
    return s


# ---------------------------------------------------------------------------------------------------------- one pass

def run(state):
    s, c = state, state["case"]
    kind, ctx = c["kind"], s["ctx"]
    if kind == "map":
        return ctx.trace_image(s["grid"], s["view"], s["freqs"], s["opts"])
    if kind == "batch":
        s["plan"].launch()
        return list(s["plan"].outputs)
    if kind == "spectrum":
        tb = ctx.trace_image(s["grid"], s["view"], s["freqs"], s["opts"])
        return {"tb": tb, "mean": ctx.disk_mean_tb(s["view"], tb)}
    if kind == "snapshot":
        grid = ctx.load_grid(*s["axes"], s["ne"], s["te"])
        tb = ctx.trace_image(grid, s["view"], s["freqs"], s["opts"])
        grid.free()
        return tb
    if kind == "tape":
        tb, _, tape = ctx.trace_image_tape(s["grid"], s["view"], s["freqs"], s["opts"])
        dne, dte = tape.backward(s["w"])
        tape.free()
        return {"tb": tb, "dne": dne, "dte": dte}
    if kind == "autograd":
        tb = rt.RayTraceFn.apply(s["ne"], s["te"], ctx, *s["axes"], s["view"], s["freqs"], s["opts"])
        dne, dte = torch.autograd.grad(tb, (s["ne"], s["te"]), s["w"])
        return {"tb": tb.detach(), "dne": dne, "dte": dte}
    if kind == "beam":
        return ctx.beam_convolve(s["view"], s["tb"], s["freqs"], c["baseline"])
    return ctx.disk_mean_tb(s["view"], s["tb"], c["radius"])


# ------------------------------------------------------------------------------------------------------- what it takes

C_PE = 4.803204712570263e-10 ** 2 / (math.pi * 9.1093837015e-28)  # f_pe^2 / n_e, CGS
R_SUN_CM = 6.957e10
# FP32 operations (FMA = 2) of one central step: 4 field evaluations of 111, the RK4 sums 60, transfer and
# termination 100; with magnification the tube area needs at least the second derivatives of the field at the three
# stage points that the separations depend on, about 60 each, with the chord's directions
FLOP_STEP = 4 * 111 + 60 + 100
FLOP_MAG = 3 * 60 + 30
# the reverse of a step: its recomputation, and about three times its operations
ADJOINT = 4


def _ray_steps(c, view, freqs):
    """Central steps of a map, from the straight entry chords cut where n_e of the background reaches the plasma
    frequency or at the inner sphere."""
    u = view.x0 + (np.arange(view.nx) + 0.5) * (view.x1 - view.x0) / view.nx
    w = view.y0 + (np.arange(view.ny) + 0.5) * (view.y1 - view.y0) / view.ny
    b = np.sqrt(u[None, :] ** 2 + w[:, None] ** 2)
    b = b[b < c["r_max"]]
    steps = 0.0
    for f in freqs:
        x = math.log10(f * f / C_PE / 4.2e4)
        rc = 4.32 / x if x > 0 else 1e9
        out = np.sqrt(c["r_max"] ** 2 - b * b)
        stop = max(min(rc, c["r_max"]), 1.0)
        inn = np.sqrt(np.maximum(stop * stop - b * b, 0.0))
        steps += float(np.where(b >= stop, 2 * out, (2 if rc > 1 else 1) * (out - inn)).sum())
    return steps / c["dtau"]


def work(case):
    c, kind = case, case["kind"]
    px = c["nx"] * c["ny"] * c["nf"]
    if kind == "beam":
        dx = 2.0 * c["extent"] / max(c["nx"], c["ny"])
        taps = sum(2 * math.ceil(4 * _sigma(f, c["baseline"], dx)) + 1 for f in _freqs(c))
        return {"bytes": 8.0 * px, "flops": 4.0 * c["nx"] * c["ny"] * taps}
    if kind == "disk":
        share = min(1.0, math.pi * c["radius"] ** 2 / (4.0 * c["extent"] ** 2))
        return {"bytes": 4.0 * px * share + 8.0 * c["nf"], "flops": px * share}
    nodes = c["n_r"] * c["n_t"] * c["n_p"]
    grid_bytes = 2.0 * nodes * (8 if c["f64"] else 4)
    if kind == "batch":
        reqs = _requests(c, 0)
        steps = sum(_ray_steps(c, v, f) for v, f in reqs)
        px = sum(v.nx * v.ny * len(f) for v, f in reqs)
    else:
        steps = _ray_steps(c, _view(c), _freqs(c))
    per = FLOP_STEP + (0 if c["mode"] == rt.RT_MAG_OFF else FLOP_MAG)
    if c["mode"] == rt.RT_TUBE:
        per = FLOP_STEP * (1 + c["nb"])
    both = kind in ("tape", "autograd")
    return {"bytes": grid_bytes * (2 if both else 1) + 4.0 * px * (2 if both else 1),
            "flops": steps * per * (1 + ADJOINT if both else 1)}


# ------------------------------------------------------------------------------------------------- the same in 64 bits

def _sigma(f, baseline, dx):
    """Beam width in pixels: FWHM = lambda / B radians at 1 AU."""
    return 2.99792458e10 / f / (baseline * 100.0) * (1.495978707e13 / R_SUN_CM) / math.sqrt(8.0 * math.log(2.0)) / dx


class _Field:
    """n_e, T_e and grad n_e of the trilinear interpolant in (r, theta, phi), float64."""

    def __init__(self, r, th, ph, ne, te):
        self.r = torch.tensor(r, device=DEV)
        self.n = ne.shape
        self.t0, self.dt = float(th[0]), float((th[-1] - th[0]) / (len(th) - 1))
        self.p0, self.dp = float(ph[0]), 2.0 * math.pi / len(ph)
        self.ne, self.te = ne.detach().double().reshape(-1), te.detach().double().reshape(-1)
        self.r_vac = float(r[-1]) * (1.0 + 1e-6)
        a = torch.arange(8, device=DEV)[:, None]
        self.da, self.db, self.dc = a // 4, a // 2 % 2, a % 2

    def __call__(self, p, want_te=False):
        n_r, n_t, n_p = self.n
        x, y, z = p[0], p[1], p[2]
        rho2 = x * x + y * y
        r2 = rho2 + z * z
        r, rho = r2.sqrt(), rho2.sqrt()
        i = (torch.searchsorted(self.r, r, right=True) - 1).clamp(0, n_r - 2)
        R = self.r[i]
        idr = 1.0 / (self.r[i + 1] - R)
        u = (r - R) * idr
        tt = (torch.atan2(rho, z) - self.t0) / self.dt
        j = tt.floor().clamp(0, n_t - 2)
        v = (tt - j).clamp(0, 1)
        tsel = ((tt > 0) & (tt < n_t - 1)).double()
        pp = torch.remainder(torch.atan2(y, x) - self.p0, 2.0 * math.pi) / self.dp
        k = pp.floor().clamp(0, n_p - 1)
        w = pp - k
        kc = (k.long() + self.dc) % n_p
        idx = ((i + self.da) * n_t + (j.long() + self.db)) * n_p + kc
        inside = (r <= self.r_vac).double()

        def lerp(vals):
            C = vals[idx].reshape(2, 2, 2, -1) * inside
            D = C[:, :, 1] - C[:, :, 0]
            A = C[:, :, 0] + w * D
            E = A[:, 1] - A[:, 0]
            B = A[:, 0] + v * E
            return B, E, D

        B, E, D = lerp(self.ne)
        fu = B[1] - B[0]
        f = B[0] + u * fu
        fv = E[0] + u * (E[1] - E[0])
        G = D[:, 0] + v * (D[:, 1] - D[:, 0])
        fw = G[0] + u * (G[1] - G[0])
        irho = torch.where(rho2 > 0, 1.0 / rho, torch.zeros_like(rho))
        a = fu * idr / r
        ft = fv * tsel / self.dt
        b = ft * z / r2 * irho
        cc = fw / self.dp * irho * irho
        g = torch.stack([(a + b) * x - cc * y, (a + b) * y + cc * x, a * z - ft * rho / r2])
        if not want_te:
            return f, g, None
        Bt, _, _ = lerp(self.te)
        return f, g, Bt[0] + u * (Bt[1] - Bt[0])


def _dot(a, b):
    return (a * b).sum(-2)


def _cross(a, b):
    return torch.stack([a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]])


def _crossing(p, dr, R, leaving):
    A, B, C = _dot(dr, dr), 2 * _dot(p, dr), _dot(p, p) - R * R
    q = (B * B - 4 * A * C).clamp(min=0).sqrt()
    return ((-B + q) / (2 * A) if leaving else (-B - q) / (2 * A)).clamp(0, 1)


def _kappa(ne, te, f2, lnf):
    ok = (ne > 0) & (te > 0)
    t = torch.where(ok, te, torch.ones_like(te))
    g = torch.where(t > 2e5, 24.5 + t.log() - lnf, 18.2 + 1.5 * t.log() - lnf)
    return torch.where(ok, 9.78e-3 / f2 * ne * ne * g / t ** 1.5, torch.zeros_like(ne))


def _trace64(c, corona, rays):
    """T_b of `rays` (list of (view, freqs)), flat in the order of their maps."""
    r, _, _, _, _ = corona
    F = _Field(*corona)
    h, nb = c["dtau"], (0 if c["mode"] == rt.RT_MAG_OFF else c["nb"])
    r_min, r_max, eta, tau_stop = float(r[0]), float(r[-1]), 0.5, 30.0
    P, O, FR = [], [], []
    for v, freqs in rays:
        cl, sl, cb, sb = math.cos(v.lon_rad), math.sin(v.lon_rad), math.cos(v.lat_rad), math.sin(v.lat_rad)
        o = torch.tensor([cb * cl, cb * sl, sb], device=DEV, dtype=torch.float64)[:, None]
        eu = torch.tensor([-sl, cl, 0.0], device=DEV, dtype=torch.float64)[:, None]
        ev = torch.tensor([-sb * cl, -sb * sl, cb], device=DEV, dtype=torch.float64)[:, None]
        q = torch.arange(v.nx * v.ny, device=DEV)
        a = v.x0 + (q % v.nx + 0.5) * ((v.x1 - v.x0) / v.nx)
        b = v.y0 + (q // v.nx + 0.5) * ((v.y1 - v.y0) / v.ny)
        d = (r_max * r_max - a * a - b * b).clamp(min=0).sqrt().double()
        for f in freqs:
            P.append(a * eu + b * ev + d * o)
            O.append(o.expand(3, q.numel()))
            FR.append(torch.full((q.numel(),), float(f), device=DEV, dtype=torch.float64))
    p, o, fr = torch.cat(P, 1).clone(), torch.cat(O, 1), torch.cat(FR)
    f2, lnf, kf = fr * fr, fr.log(), -C_PE / (2.0 * fr * fr)
    n2 = 1.0 - C_PE * F(p)[0] / f2
    k = -n2.clamp(min=0).sqrt() * o
    z = torch.zeros_like(fr)
    active = n2 > 0  # every line of sight of these views meets the outer sphere
    first = torch.ones_like(active)
    S = {"p": p, "k": k.clone(), "tb": z.clone(), "tau": z.clone(), "lns": z.clone(), "kap": z.clone(),
         "te": z.clone(), "active": active, "first": first}

    def step():
        p, k, live = S["p"], S["k"], S["active"]
        ne, g1, te = F(p, True)
        a1 = kf * g1
        a2 = kf * F(p + h / 2 * k)[1]
        a3 = kf * F(p + h / 2 * (k + h / 2 * a1))[1]
        a4 = kf * F(p + h * (k + h / 2 * a2))[1]
        G0 = a1 + a2 + a3
        kap = _kappa(ne, te, f2, lnf)
        on = live & ~S["first"]
        dt = 0.5 * (S["kap"] + kap) * h * R_SUN_CM
        w = 0.5 * (S["te"] + te) * -torch.expm1(-dt) * torch.exp(S["lns"] - S["tau"])
        S["tb"].add_(torch.where(on, w, z))
        S["tau"].add_(torch.where(on, dt, z))
        live = live & ~(on & (S["tau"] >= tau_stop))
        dr = h * k + h * h / 6 * G0
        kn = k + h / 6 * (a1 + 2 * a2 + 2 * a3 + a4)
        rn = p + dr
        rr = _dot(rn, rn)
        hit = live & (rr < r_min * r_min)
        out = live & ~hit & (rr > r_max * r_max) & (_dot(rn, kn) > 0)
        if nb:
            ds = _dot(dr, dr).sqrt()
            t = dr / ds
            use_z = t[2].abs() <= 0.9
            zero = torch.zeros_like(ds)
            e1 = torch.where(use_z, torch.stack([-t[1], t[0], zero]), torch.stack([t[2], zero, -t[0]]))
            e1 = e1 / _dot(e1, e1).sqrt()
            e2 = _cross(t, e1)
            eps = eta * ds
            s2 = math.sqrt(0.5)
            dirs = [e1, e2] if nb < 8 else [e1, e2, s2 * (e1 + e2), s2 * (e2 - e1)]
            seeds = dirs if nb == 2 else [x for e in dirs for x in (e, -e)]
            m = len(seeds)
            q = torch.cat([p + eps * e for e in seeds], 1)
            kk, kfm = k.repeat(1, m), kf.repeat(m)
            b1 = kfm * F(q)[1]
            G = b1 + kfm * F(q + h / 2 * kk)[1] + kfm * F(q + h / 2 * (kk + h / 2 * b1))[1]
            G = G.reshape(3, m, -1)
            if nb == 2:
                D = [h * h / 6 / eps * (G[:, j] - G0) for j in range(2)]
            else:
                D = [h * h / 12 / eps * (G[:, 2 * j] - G[:, 2 * j + 1]) for j in range(m // 2)]

            def mag(d1, d2, x1, x2):
                return (1.0 + _dot(d1, x1) + _dot(d2, x2) + _dot(t, _cross(d1, d2))).abs()

            M = mag(D[0], D[1], e1, e2)
            if nb == 8:
                M = 0.5 * (M + mag(D[2], D[3], dirs[2], dirs[3]))
            S["lns"].add_(torch.where(live, M.log(), z))
        # the clipped last segment and the boundary term
        al = torch.where(hit, _crossing(p, dr, r_min, False), _crossing(p, dr, r_max, True))
        nee, _, tee = F(p + al * dr, True)
        dte = 0.5 * (kap + _kappa(nee, tee, f2, lnf)) * h * R_SUN_CM * al
        end = hit | out
        w = 0.5 * (te + tee) * -torch.expm1(-dte) * torch.exp(S["lns"] - S["tau"])
        S["tb"].add_(torch.where(end, w, z))
        S["tau"].add_(torch.where(end, dte, z))
        S["tb"].add_(torch.where(hit, tee * torch.exp(S["lns"] - S["tau"]), z))
        live = live & ~end
        S["p"].copy_(torch.where(live, rn, p))
        S["k"].copy_(torch.where(live, kn, k))
        S["kap"].copy_(kap)
        S["te"].copy_(te)
        S["active"].copy_(live)
        S["first"].fill_(False)

    step()
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        step()
    torch.cuda.current_stream().wait_stream(side)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        step()
    for _ in range(int(40.0 * r_max / h) // 128 + 1):
        for _ in range(128):
            graph.replay()
        if not bool(S["active"].any()):
            break
    return S["tb"]


# what _trace64 does within about 20 seconds: it takes some 3 milliseconds a step, whatever the rays, up to these
MOST_STEPS, MOST_RAYS = 4200, 2.4e5


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "beam":
        tb, dx = _maps(c, seed).double(), 2.0 * c["extent"] / max(c["nx"], c["ny"])
        out = torch.empty_like(tb)
        for i, f in enumerate(_freqs(c)):
            sg = _sigma(f, c["baseline"], dx)
            hw = math.ceil(4.0 * sg)

            def band(n):
                d = torch.arange(n, device=DEV, dtype=torch.float64)
                d = d[:, None] - d[None, :]
                e = torch.arange(-hw, hw + 1, device=DEV, dtype=torch.float64)
                return torch.exp(-d * d / (2 * sg * sg)) * (d.abs() <= hw) / torch.exp(-e * e / (2 * sg * sg)).sum()
            out[i] = band(c["ny"]) @ tb[i] @ band(c["nx"])
        return out
    v = _view(c)

    def mean(tb, radius):
        u = v.x0 + (torch.arange(v.nx, device=DEV, dtype=torch.float64) + 0.5) * ((v.x1 - v.x0) / v.nx)
        w = v.y0 + (torch.arange(v.ny, device=DEV, dtype=torch.float64) + 0.5) * ((v.y1 - v.y0) / v.ny)
        inside = (u[None, :] ** 2 + w[:, None] ** 2) < radius * radius
        n = int(inside.sum())
        return tb.double()[:, inside].sum(1) / n if n else torch.zeros(c["nf"], dtype=torch.float64, device=DEV)

    if kind == "disk":
        return mean(_maps(c, seed), c["radius"])
    # the reverse sweep and the rays of tube mode and of the global corona (30000 steps each) take too long here
    if kind in ("tape", "autograd", "snapshot") or c["mode"] == rt.RT_TUBE or c["corona"] == "global":
        return None
    rays = _requests(c, seed) if kind == "batch" else [(v, _freqs(c))]
    n = sum(a.nx * a.ny * len(f) for a, f in rays) * (1 if c["mode"] == rt.RT_MAG_OFF else max(1.0, c["nb"] / 4.0))
    if n > MOST_RAYS or 2.0 * c["r_max"] / c["dtau"] > MOST_STEPS:
        return None
    tb = _trace64(c, _corona(c, seed), rays)
    if kind == "batch":
        out, at = [], 0
        for a, f in rays:
            m = a.nx * a.ny * len(f)
            out.append(tb[at:at + m].reshape(len(f), a.ny, a.nx))
            at += m
        return out
    tb = tb.reshape(c["nf"], c["ny"], c["nx"])
    return {"tb": tb, "mean": mean(tb, 0.5)} if kind == "spectrum" else tb
