"""Timed cases of the visibility simulator: what its users have it compute, from one small slice to the
whole polarised 350-antenna simulation, through the public entry points (Plan, Batch).

A case is a dict of plain values:

  mode      "run":    a resident plan and sky, visibilities into a device buffer (Plan.run)
            "fresh":  a new sky from host memory every pass and the result back in pinned host memory
                      (Plan.set_sky, Plan.run), as a calibration or Monte-Carlo loop does
            "ragged": independent single-slice problems of many sizes replayed as one CUDA graph (Batch)
            "tick":   one tick of a server: a block of channels of one time from each of three resident
                      plans, added to a Batch and executed plainly
  radius    rings of the hexagonal array, 14.6 m spacing (3: 37, 6: 127, 10: 331 antennas); keep > 0 cuts it
            to that many antennas
  jitter    antennas moved by 0.4 m horizontally, so that the array is not a lattice (every baseline is its
            own target); height: 5 cm vertical scatter
  channels, times, points, nside (HEALPix pixels of the diffuse map as sources; 0: none)
  pol       Stokes IQUV and four products, else one;  fp64, eps: precision and tolerance
  route     Plan's transform argument;  beam: "gauss", "airy", "grid" (numerical samples) or "mixed" (two
            dish sizes and a numerical beam dealt over the antennas)
  slices    ragged: how many problems;  mix: which draw of their sizes
"""
import math

import numpy as np
import torch

from paper_2506_02130_gb300 import fv, workloads as W

C_LIGHT = 299792458.0
BASE = {"mode": "run", "radius": 6, "keep": 0, "jitter": False, "height": False, "channels": 1, "times": 1,
        "points": 1000, "nside": 0, "pol": False, "fp64": False, "eps": 1e-6, "route": "auto", "beam": "gauss",
        "slices": 0, "mix": 0}


def _case(name=None, **kw):
    c = dict(BASE, **kw)
    return c if name is None else dict(c, name=name)


def listed():
    hex127 = dict(radius=6, height=True, points=20000, nside=64)
    hex350 = dict(radius=11, keep=350, points=100000, nside=256, pol=True, beam="airy", route="type3")
    return [
        # the first thing a user runs, and the inner call of a fitting loop: one slice of a small array in FP64
        _case("small_fp64", radius=3, fp64=True, eps=1e-10),
        # one snapshot of the large array: a single slice, where nothing overlaps it
        _case("snapshot_350_pol", **hex350),
        # a server's tick: 32, 16 and 6 channels of one time of three resident problems
        _case("tick", mode="tick", channels=32),
        # a simulation of a lattice array with height scatter, route left to the plan
        _case("hex127_auto", channels=64, times=10, **hex127),
        # the same through the general-array path, a single precision for sampled maps
        _case("hex127_type3", channels=64, times=10, route="type3", **hex127),
        # reference-quality results: every step in FP64
        _case("hex127_fp64", channels=8, times=2, route="type3", fp64=True, eps=1e-11, **hex127),
        # all channels of a time through one spectral basis
        _case("hex127_basis", channels=64, times=10, route="basis", **hex127),
        # a general polarised array: neither coplanar nor on a lattice, every baseline a target of its own
        _case("jitter127_pol", channels=16, times=2, radius=6, jitter=True, height=True, points=20000, nside=64,
              pol=True, beam="airy"),
        # antennas with different beams, one of them numerical: one transform per pair of beams
        _case("mixed_beams_61", channels=16, times=4, radius=4, points=5000, nside=32, beam="mixed", route="type3"),
        # many small independent problems of both precisions at once
        _case("ragged", mode="ragged", slices=48),
        # a new polarised sky every pass, host to host
        _case("fresh_350_pol", **dict(hex350, mode="fresh", channels=6)),
        # the full polarised simulation, the largest call
        _case("hex350_pol", channels=256, times=4, **hex350),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _n_src(c):
    return c["points"] + 12 * c["nside"] ** 2


def draw(rng):
    kind = rng.choice(["small", "lattice", "general", "fp64", "basis", "jitter", "beams", "pol", "fresh", "ragged",
                       "tick"])
    if kind == "tick":
        return _case(mode="tick", channels=rng.randint(8, 40))
    if kind == "ragged":
        return _case(mode="ragged", slices=int(_log(rng, 6, 56)), mix=rng.randint(1, 1000))
    c = _case(radius=rng.randint(3, 10), channels=int(_log(rng, 1, 257)), times=rng.randint(1, 20),
              points=int(_log(rng, 1000, 200001)), nside=rng.choice([0, 0, 16, 32, 64, 128]))
    if kind == "small":
        c.update(radius=rng.randint(3, 5), channels=rng.randint(1, 4), times=1, nside=0, fp64=rng.random() < 0.5,
                 points=int(_log(rng, 300, 5000)), eps=rng.choice([1e-6, 1e-5]))
        if c["fp64"]:
            c["eps"] = rng.choice([1e-10, 1e-9, 1e-7])
    elif kind == "lattice":
        c["height"] = rng.random() < 0.5
    elif kind == "general":
        c.update(route="type3", height=rng.random() < 0.7, eps=rng.choice([1e-6, 1e-6, 1e-5]))
    elif kind == "fp64":
        c.update(route=rng.choice(["type3", "auto"]), fp64=True, eps=rng.choice([1e-11, 1e-10, 1e-8]),
                 height=rng.random() < 0.5, radius=rng.randint(3, 8))
    elif kind == "basis":
        c.update(route="basis", height=rng.random() < 0.7, channels=rng.randint(16, 96), times=rng.randint(1, 10),
                 radius=rng.randint(3, 6))
    elif kind == "jitter":
        c.update(jitter=True, height=rng.random() < 0.6, pol=rng.random() < 0.5, radius=rng.randint(3, 6),
                 beam=rng.choice(["gauss", "airy", "grid"]))
    elif kind == "beams":
        c.update(beam="mixed", route=rng.choice(["type3", "auto"]), radius=rng.randint(3, 5))
    elif kind == "pol":
        c.update(radius=rng.randint(5, 11), pol=True, beam=rng.choice(["airy", "gauss", "grid"]),
                 route=rng.choice(["type3", "auto"]), nside=rng.choice([64, 128, 256]))
    else:
        c.update(mode="fresh", pol=rng.random() < 0.5, beam="airy", times=1, channels=int(_log(rng, 1, 33)))
    # keep a drawn case well below the largest listed one: fewer times, then fewer channels
    units = (0.3e6 + _n_src(c)) * (4 if c["pol"] else 1) * (4 if c["beam"] == "mixed" else 1) * (45 if c["fp64"] else 1)
    most = max(1, int(1.2e9 / units))
    c["times"] = min(c["times"], max(1, most // c["channels"]))
    c["channels"] = min(c["channels"], most)
    if c["mode"] == "fresh":
        c["channels"] = min(c["channels"], max(1, int(8e6 / (_n_src(c) * (4 if c["pol"] else 1)))))
    return c


# ---------------------------------------------------------------------------------------------- inputs
_stream = None
_device = "cuda"


def _the_stream():
    """A program's one compute stream."""
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    return _stream


def _diffuse(g, n, d):
    """A smooth unit-variance field at the directions n [n][3]: random plane waves with a falling spectrum."""
    k = torch.randn(48, 3, generator=g, device=_device, dtype=torch.float64)
    k *= (2.0 + 30.0 * torch.rand(48, 1, generator=g, device=_device, dtype=torch.float64) ** 2)
    a = torch.randn(48, generator=g, device=_device, dtype=torch.float64) / k.norm(dim=1).clamp_min(1.0) ** 0.75
    ph = 2 * math.pi * torch.rand(48, generator=g, device=_device, dtype=torch.float64)
    f = torch.cos(n @ k.T + ph) @ a
    return ((f - f.mean()) / f.std()).to(d)


def _sky(points, nside, pol, freqs, g, d, hemisphere=None):
    """(ra, dec, flux [stokes][source][channel]) on the GPU: power-law point sources, uniform on the sphere (or
    above the horizon at hemisphere = (lst, latitude)), and the pixels of a diffuse map; a tenth polarised."""
    f64 = dict(device=_device, dtype=torch.float64)
    u = torch.rand(4, max(points, 1), generator=g, **f64)[:, :points]
    if hemisphere is None:
        ra, dec = 2 * math.pi * u[0], torch.asin(2 * u[1] - 1)
    else:
        r, s = W.visible_hemisphere(points, np.random.default_rng(int(u.sum() * 1e6) if points else 0), *hemisphere)
        ra, dec = torch.as_tensor(r, device=_device), torch.as_tensor(s, device=_device)
    amp = torch.exp(math.log(0.1) + u[2] * math.log(100.0))
    index = -0.8 + 0.2 * torch.randn(points, generator=g, **f64)
    if nside:
        pr, pd = (torch.as_tensor(v, device=_device) for v in W.healpix_radec(nside))
        n = torch.stack([torch.cos(pd) * torch.cos(pr), torch.cos(pd) * torch.sin(pr), torch.sin(pd)], dim=1)
        field = _diffuse(g, n, torch.float64)
        amp = torch.cat([amp, 1e3 * torch.exp(0.5 * field - 0.125) * W.healpix_pixel_area(nside)])
        index = torch.cat([index, -2.5 + 0.1 * torch.randn(len(pr), generator=g, **f64)])
        ra, dec = torch.cat([ra, pr]), torch.cat([dec, pd])
    x = torch.log(torch.as_tensor(freqs, device=_device) / 150e6).to(d)
    spec = torch.exp(index.to(d)[:, None] * x[None, :]) * amp.to(d)[:, None]
    if not pol:
        return ra.cpu().numpy(), dec.cpu().numpy(), spec[None].contiguous()
    flux = torch.zeros((4,) + tuple(spec.shape), device=_device, dtype=d)
    q = 0.1 * torch.randn(2, len(amp), generator=g, **f64).to(d)
    flux[0] = spec
    torch.mul(spec, q[0][:, None], out=flux[1])
    torch.mul(spec, q[1][:, None], out=flux[2])
    return ra.cpu().numpy(), dec.cpu().numpy(), flux


def _beams(c, freqs):
    """(plan beam kind, parameters, per-antenna beams or None, gridded samples by beam index)."""
    samples = W.grid_beam(freqs, 61, 36, math.radians(20.0), 150e6, ellipticity=0.2)
    if c["beam"] == "airy":
        return "airy", (14.0,), None, {}
    if c["beam"] == "grid":
        return "uniform", (), None, {-1: samples}
    if c["beam"] == "mixed":
        return "gauss", W.GAUSS_FWHM_150, [("gauss", W.GAUSS_FWHM_150), ("airy", (9.0,)), ("grid", ())], {2: samples}
    return "gauss", W.GAUSS_FWHM_150, None, {}


def _problem(c, seed):
    rng = np.random.default_rng([seed, 7])
    g = torch.Generator(device=_device)
    g.manual_seed(1000003 * seed + 17)
    ant = W.hex_array(c["radius"], n_keep=c["keep"] or None)
    if c["jitter"]:
        ant[:, :2] += rng.normal(0.0, 0.4, (len(ant), 2))
    if c["height"]:
        ant[:, 2] = rng.normal(0.0, 0.05, len(ant))
    freqs = np.array([150e6]) if c["channels"] == 1 else W.channel_centres(c["channels"])
    lst0 = rng.uniform(0, 2 * np.pi)
    lsts = W.lst_grid(c["times"], 10.7, lst0)
    up = (lst0, W.HERA_LATITUDE_RAD) if c["nside"] == 0 and c["points"] <= 1000 and c["times"] == 1 else None
    ra, dec, flux = _sky(c["points"], c["nside"], c["pol"], freqs, g, torch.float64 if c["fp64"] else torch.float32,
                         up)
    kind, param, beams, grids = _beams(c, freqs)
    boa = rng.integers(0, 3, len(ant)) if beams else None
    return dict(c=c, ant=ant, freqs=freqs, lsts=lsts, ra=ra, dec=dec, flux=flux, kind=kind, param=param, beams=beams,
                grids=grids, boa=boa)


def _ragged(c, seed):
    """Single-slice problems: hexagons of 37 to 331 antennas, 1e3 to 5e5 sources, both precisions (the sizes
    follow from the case, the frequencies, times and skies from the seed)."""
    size, rng = np.random.default_rng([c["mix"], 11]), np.random.default_rng([seed, 11])
    out = []
    for k in range(c["slices"]):
        fp64 = size.random() < 0.5
        one = dict(BASE, radius=int(size.integers(3, 11)),
                   points=int(math.exp(size.uniform(math.log(1e3), math.log(5e5)))),
                   fp64=bool(fp64), eps=1e-10 if fp64 else 1e-6)
        p = _problem(one, seed * 64 + k)
        nu = np.array([rng.uniform(100e6, 200e6)])
        p["flux"] = p["flux"] * float((nu[0] / 150e6) ** -0.8)
        p["freqs"] = nu
        out.append(p)
    return out


def _tick(c, seed):
    """The resident problems of a server and the (channel, time) block that a tick takes from each."""
    n = c["channels"]
    hex350 = dict(radius=11, keep=350, points=100000, nside=256, pol=True, beam="airy")
    probs = [_problem(dict(BASE, radius=3, points=1001, channels=n, times=4), seed),
             _problem(dict(BASE, height=True, points=20000, nside=64, channels=n, times=4), seed + 1),
             _problem(dict(BASE, channels=n, times=4, **hex350), seed + 2)]
    rng = np.random.default_rng([seed, 13])
    blocks = []
    for m in (n, max(1, n // 2), max(1, 6 * n // 32)):
        f0, t0 = int(rng.integers(0, n - m + 1)), int(rng.integers(0, 4))
        blocks.append(((f0, f0 + m), (t0, t0 + 1)))
    return probs, blocks


def _plan(p):
    c = p["c"]
    plan = fv.Plan.create(p["freqs"], p["lsts"], W.HERA_LATITUDE_RAD, p["kind"], p["param"],
                          fv.FV_FP64 if c["fp64"] else fv.FV_MIXED, c["eps"], c["pol"],
                          stream=_the_stream().cuda_stream, transform=c["route"])
    plan.set_array(p["ant"])
    if p["beams"]:
        plan.set_beams(p["beams"], p["boa"], p["grids"])
    elif p["grids"]:
        plan.set_beam_grid(-1, p["grids"][-1])
    return plan


def _out(p, shape, **kw):
    return torch.empty(shape, dtype=torch.complex128 if p["c"]["fp64"] else torch.complex64, **kw)


def prepare(case, seed):
    c = dict(BASE, **case)
    if c["mode"] == "fresh":
        p = _problem(c, seed)
        return dict(mode="fresh", plan=_plan(p), ra=p["ra"], dec=p["dec"], flux=p["flux"].cpu().pin_memory().numpy(),
                    out=[_out(p, (c["channels"], c["times"], len(p["ant"]) * (len(p["ant"]) - 1) // 2,
                                  4 if c["pol"] else 1), pin_memory=True).numpy()])
    if c["mode"] in ("ragged", "tick"):
        probs, blocks = (_ragged(c, seed), None) if c["mode"] == "ragged" else _tick(c, seed)
        plans, outs = [], []
        for k, p in enumerate(probs):
            plan = _plan(p)
            torch.cuda.synchronize()
            plan.set_sky(p["ra"], p["dec"], p["flux"].cpu().numpy() if c["mode"] == "ragged" else p["flux"])
            shape = plan.out_shape
            if blocks:
                (f0, f1), (t0, t1) = blocks[k]
                shape = (f1 - f0, t1 - t0) + shape[2:]
            plans.append(plan)
            outs.append(_out(p, shape, device=_device))
        torch.cuda.synchronize()
        batch = fv.Batch(stream=_the_stream().cuda_stream)
        if not blocks:
            for plan, o in zip(plans, outs):
                batch.add(plan, o)
        return dict(mode=c["mode"], batch=batch, plans=plans, out=outs, blocks=blocks)
    p = _problem(c, seed)
    plan = _plan(p)
    torch.cuda.synchronize()
    plan.set_sky(p["ra"], p["dec"], p["flux"])
    return dict(mode="run", plan=plan, out=[_out(p, plan.out_shape, device=_device)])


def run(state):
    if state["mode"] == "run":
        state["plan"].run(state["out"][0])
    elif state["mode"] == "fresh":
        state["plan"].set_sky(state["ra"], state["dec"], state["flux"])
        state["plan"].run(state["out"][0])
    elif state["mode"] == "ragged":
        state["batch"].execute(use_graph=True)
    else:
        b = state["batch"]
        b.clear()
        for plan, o, (f, t) in zip(state["plans"], state["out"], state["blocks"]):
            b.add(plan, o, t, f, window=(f[0], t[0], t[1] - t[0]))
        b.execute()
    return state["out"]


# ---------------------------------------------------------------------------------------------- work
def _work(c, n_slices):
    """Sources above the horizon (half of them) read once with their fluxes and spread over w x w cells per product,
    an oversampled transform of the array's extent, w x w cells read per unique baseline, the result written."""
    w = math.ceil(math.log10(1 / c["eps"])) + 1
    es = 8 if c["fp64"] else 4
    npol, n_src = 4 if c["pol"] else 1, _n_src(c)
    n_ant = c["keep"] or 3 * c["radius"] * (c["radius"] + 1) + 1
    n_bl = n_ant * (n_ant - 1) // 2
    n_u = n_bl if c["jitter"] or c["height"] else 3 * (2 * c["radius"]) * (2 * c["radius"] + 1) // 2
    X = 2 * math.pi * 150e6 / C_LIGHT * 14.6 * 2 * c["radius"]
    cells = (2 * X / math.pi * 2 + w) * (X / math.pi * 2 + w)
    nvis = 0.5 * n_src
    bytes_ = nvis * (24 + npol * es * n_slices) + n_slices * n_bl * npol * 2 * es
    flops = n_slices * npol * (4 * nvis * w * w + 5 * cells * math.log2(cells) + 4 * n_u * w * w)
    return bytes_, flops


def work(case):
    c = dict(BASE, **case)
    if c["mode"] == "ragged":
        parts = [(dict(BASE, radius=6, points=80000, fp64=bool(k), eps=1e-10 if k else 1e-6), c["slices"] / 2)
                 for k in (0, 1)]
    elif c["mode"] == "tick":
        n = c["channels"]
        parts = [(dict(BASE, radius=3), n), (dict(BASE, height=True, points=20000, nside=64), n / 2),
                 (dict(BASE, radius=11, keep=350, points=100000, nside=256, pol=True), max(1, 6 * n // 32))]
    else:
        parts = [(c, c["channels"] * c["times"])]
    got = [_work(*p) for p in parts]
    return {"bytes": sum(g[0] for g in got), "flops": sum(g[1] for g in got)}


# ---------------------------------------------------------------------------------------------- 64-bit values
def _grid_voltage(samples, f, s):
    """Bilinear interpolation of one channel's samples in zenith angle and azimuth (east of north)."""
    t = torch.as_tensor(samples[f], device=_device)
    nt, npix = t.shape
    u = torch.atan2(torch.hypot(s[0], s[1]), s[2]) / ((math.pi / 2) / (nt - 1))
    v = torch.remainder(torch.atan2(s[0], s[1]), 2 * math.pi) / (2 * math.pi / npix)
    i = u.floor().clamp(0, nt - 2).long()
    j = v.floor().long()
    a, b = u - i, v - j
    j0, j1 = j % npix, (j + 1) % npix
    return (1 - a) * ((1 - b) * t[i, j0] + b * t[i, j1]) + a * ((1 - b) * t[i + 1, j0] + b * t[i + 1, j1])


def _voltage(kind, param, samples, f, nu, s):
    rho = torch.hypot(s[0], s[1])
    if kind == "grid":
        return _grid_voltage(samples, f, s)
    if kind == "gauss":
        fwhm = param[0] * param[1] / nu
        return torch.exp(-2 * math.log(2) * torch.atan2(rho, s[2]) ** 2 / fwhm ** 2)
    if kind == "airy":
        x = math.pi * param[0] * nu / C_LIGHT * rho
        return torch.where(x < 1e-8, torch.ones_like(x), 2 * torch.special.bessel_j1(x) / x.clamp_min(1e-300))
    return torch.ones_like(rho)


def _exact_vis(p, f_range=None, t_range=None):
    """The direct sum over the sources above the horizon, [channel][time][baseline][product], from antenna phasors."""
    c = p["c"]
    nf, nt, n_ant = len(p["freqs"]), len(p["lsts"]), len(p["ant"])
    f_range, t_range = f_range or (0, nf), t_range or (0, nt)
    ij = torch.triu_indices(n_ant, n_ant, 1, device=_device)
    npol = 4 if c["pol"] else 1
    out = torch.zeros((f_range[1] - f_range[0], t_range[1] - t_range[0], ij.shape[1], npol), device=_device,
                      dtype=torch.complex128)
    ra, dec = torch.as_tensor(p["ra"], device=_device), torch.as_tensor(p["dec"], device=_device)
    e = torch.stack([torch.cos(dec) * torch.cos(ra), torch.cos(dec) * torch.sin(ra), torch.sin(dec)])
    ant = torch.as_tensor(p["ant"], device=_device)
    beams = p["beams"] or [("grid" if -1 in p["grids"] else p["kind"], p["param"])]
    sl, cl = math.sin(W.HERA_LATITUDE_RAD), math.cos(W.HERA_LATITUDE_RAD)
    for t in range(*t_range):
        st, ct = math.sin(p["lsts"][t]), math.cos(p["lsts"][t])
        R = torch.tensor([[-st, ct, 0.0], [-sl * ct, -sl * st, cl], [cl * ct, cl * st, sl]], device=_device,
                         dtype=torch.float64)
        s = R @ e
        up = (s[2] > 0).nonzero()[:, 0]
        for part in up.split(131072):
            sv = s[:, part]
            proj = ant @ sv
            rho = torch.hypot(sv[0], sv[1])
            ca = torch.where(rho > 0, sv[1] / rho.clamp_min(1e-300), torch.ones_like(rho))
            sa = torch.where(rho > 0, sv[0] / rho.clamp_min(1e-300), torch.zeros_like(rho))
            c2, s2 = ca * ca - sa * sa, 2 * ca * sa
            for f in range(*f_range):
                nu = float(p["freqs"][f])
                cyc = proj * (nu / C_LIGHT)
                F = torch.polar(torch.ones_like(cyc), -2 * math.pi * (cyc - cyc.round()))
                A = [_voltage(k, q, p["grids"].get(b if p["beams"] else -1), f, nu, sv)
                     for b, (k, q) in enumerate(beams)]
                F = F * (torch.stack(A)[torch.as_tensor(p["boa"], device=_device)] if p["beams"] else A[0])
                I = p["flux"][:, part, f].double()
                Fh = F.conj().T
                if npol == 1:
                    prod = [(F * I[0]) @ Fh]
                else:
                    Qr, Ur = I[1] * c2 - I[2] * s2, I[1] * s2 + I[2] * c2
                    v01 = (F * torch.complex(Ur, I[3])) @ Fh
                    prod = [(F * (I[0] + Qr)) @ Fh, v01, v01.conj().T, (F * (I[0] - Qr)) @ Fh]
                for q, v in enumerate(prod):
                    out[f - f_range[0], t - t_range[0], :, q] += v[ij[0], ij[1]]
    return out


def exact(case, seed):
    c = dict(BASE, **case)
    if c["mode"] == "ragged":
        return [_exact_vis(p) for p in _ragged(c, seed)]
    if c["mode"] == "tick":
        probs, blocks = _tick(c, seed)
        return [_exact_vis(p, f, t) for p, (f, t) in zip(probs, blocks)]
    n_ant = c["keep"] or 3 * c["radius"] * (c["radius"] + 1) + 1
    cost = c["channels"] * c["times"] * 0.5 * _n_src(c) * n_ant * (8 * n_ant * (3 if c["pol"] else 1) + 800)
    if cost > 1.2e13:           # about 15 seconds
        return None
    return [_exact_vis(_problem(c, seed))]
