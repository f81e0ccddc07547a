"""Performance cases of the HVOX transforms: what a user of this library has it do.

A case names a sky (a HEALPix cap around the field centre, or a few pixels of interest), an
antenna layout (baselines of all antenna pairs), a tolerance and the calls made. The sizes are
those of the library's workloads (the LOFAR-like and SKA-Low-like configurations, the telescope
radius sweep, the sparse sky, the served request streams) and of its tests. Antennas, sky and
visibilities are drawn from the seed.

Fields of a case:
  api      plan: Plan.synthesize / Plan.analyze; batch: synthesize_batch / analyze_batch over
           several plans; noalloc: direct_synthesize_noalloc
  call     predict (sky -> vis), image (vis -> sky), step (both, one after the other)
  layout   disk (uniform), log (log-uniform radii), core (dense core and log-uniform arms),
           annuli (the radius sweep's rings); n_ant antennas, wavelength lam, n_times hour angles
           step_deg apart, n_chan channels, the first n_vis baselines (0: all), those with
           |(u, v)| <= uv_max only (0: all)
  sky      the first n_pix RING pixels at nside (n_pix 0: the cap of cap_deg); groups > 0:
           n_pix pixels in that many compact groups of the cap instead
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2306_06007_gb300 as hvox

# --------------------------------------------------------------------------- the cases


def _case(name, **kw):
    c = {"name": name, "api": "plan", "call": "step", "eps": 1e-6, "isign": -1, "weights": False, "ntrans": 1,
         "complex": False, "threshold": 0.0, "layout": "log", "n_ant": 100, "r_min_m": 50.0, "r_max_m": 100e3,
         "sigma_z_m": 10.0, "lat": 52.9, "lam": 2.0, "lam_max": 2.0, "n_times": 1, "step_deg": 15.0, "n_chan": 1,
         "n_vis": 0, "uv_max": 0.0, "nside": 64, "cap_deg": 40.0, "n_pix": 0, "groups": 0, "count": 1}
    assert not set(kw) - set(c), set(kw) - set(c)
    c.update(kw)
    return c


def _lofar(name, **kw):
    base = dict(layout="log", n_ant=300, r_min_m=50.0, r_max_m=100e3, sigma_z_m=20.0, lat=52.9, lam=1.8, lam_max=2.2,
                n_times=4, step_deg=15.0, n_chan=8, nside=256, cap_deg=30.0)
    base.update(kw)
    return _case(name, **base)


def _ska(name, **kw):
    base = dict(layout="core", n_ant=512, r_min_m=1e3, r_max_m=65e3, sigma_z_m=5.0, lat=-26.7, step_deg=3.75, nside=1024,
                cap_deg=40.0)
    base.update(kw)
    return _case(name, **base)


# antennas within a radius (km) of the sweep's layout: cumulative counts of its rings
_EDGES_KM = (0.0, 0.1, 0.3, 1.0, 3.0, 10.0, 30.0, 100.0)
_COUNTS = (24, 138, 275, 108, 145, 136, 62)


def _sweep(name, radius_km, n_pix, **kw):
    base = dict(layout="annuli", n_ant=sum(_COUNTS), r_max_m=radius_km * 1e3, sigma_z_m=5.0, lat=-26.7,
                nside=int(math.ceil(4.1 * radius_km * 1e3 / 2.0)), cap_deg=90.0, n_pix=n_pix)
    base.update(kw)
    return _case(name, **base)


def _served(name, layout, n_pix, n_vis, **kw):
    base = dict(layout=layout, n_pix=n_pix, n_vis=n_vis, nside=0, threshold=0.1)
    if layout == "log":
        base.update(n_ant=300, sigma_z_m=20.0, lat=52.9, step_deg=15.0)
    else:
        base.update(n_ant=512, r_min_m=1e3, r_max_m=65e3, sigma_z_m=5.0, lat=-26.7, step_deg=3.75)
    base.update(kw)
    return _case(name, **base)


def _core_count(uv_max, n_times):
    """Baselines with |(u, v)| <= uv_max to take: 85 % of those of the core's 307 antennas (differences of Gaussians), a
    count that every draw of the antennas has."""
    return int(0.85 * n_times * 307 * 306 / 2 * (1.0 - math.exp(-uv_max ** 2 / 500.0 ** 2)))


def listed():
    return [
        # the smallest request of a served stream: launches and latency
        _served("served_1k_f32", "core", 1000, 1000, eps=1e-4, call="predict"),
        # a large request of the small stream, the tolerance of precise imaging, ragged sizes
        _served("served_30k_df", "log", 29989, 9973, eps=1e-9, call="image", weights=True, isign=1),
        # a server's admission of eight requests of mixed tolerances in one batched call
        _served("served_batch_8", "core", 30000, 30000, eps=0.0, api="batch", call="predict", count=8),
        # a calibration solver predicting a source catalogue every iteration, allocating nothing
        _case("calibration_predict", api="noalloc", call="predict", layout="disk", n_ant=300, r_max_m=2000.0,
              n_pix=3001, nside=0, cap_deg=35.0),
        # a few pixels of interest in a wide field: long sums on one side only
        _sweep("sparse_sky", 10.0, 500, groups=5),
        # the LOFAR-like configuration at the tolerance of precise imaging: direct sums at FP64 accuracy
        _lofar("lofar_1e-9", eps=1e-9),
        # the same at single precision: direct sums and NUFFT sub-problems of the short baselines
        _lofar("lofar_1e-6", eps=1e-6),
        # one snapshot of the SKA-Low-like configuration: dense core by NUFFT, outer baselines direct
        _ska("ska_snapshot_1e-6", eps=1e-6, call="predict"),
        # the radius sweep: one NUFFT sub-problem; two stacked images (polarisations) with weights
        _sweep("radius_1km_1e-6_x2", 1.0, 130_000, eps=1e-6, ntrans=2, weights=True),
        _sweep("radius_3km_1e-6", 3.0, 810_000, eps=1e-6),
        _sweep("radius_3km_1e-9", 3.0, 810_000, eps=1e-9),
        # dense-core study: many NUFFT sub-problems in waves, a coarse tolerance
        _ska("dense_core_1e-4", eps=1e-4, n_times=8, uv_max=500.0, n_vis=_core_count(500.0, 8), nside=512),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["served", "served", "batch", "noalloc", "lofar", "ska", "sweep", "sweep", "sparse", "core"])
    eps = rng.choice([1e-4, 1e-6, 1e-9])
    call = rng.choice(["predict", "image"])
    opt = dict(weights=rng.random() < 0.5, isign=rng.choice([-1, 1]))
    if kind == "served":
        c = _served("", rng.choice(["log", "core"]), _log_int(rng, 1e3, 2e5), _log_int(rng, 1e3, 2e5), eps=eps, call=call,
                    **opt)
    elif kind == "batch":
        c = _served("", rng.choice(["log", "core"]), _log_int(rng, 3e3, 3e4), _log_int(rng, 3e3, 3e4), eps=0.0, call=call,
                    api="batch", count=rng.randint(2, 12))
    elif kind == "noalloc":
        c = _case("", api="noalloc", call="predict", layout="disk", r_max_m=rng.uniform(500.0, 5000.0),
                  n_ant=_log_int(rng, 40, 600), n_pix=_log_int(rng, 50, 3e4), nside=0, cap_deg=35.0, isign=opt["isign"])
    elif kind == "lofar":
        c = _lofar("", eps=rng.choice([1e-5, 1e-6, 1e-9]), call=call, n_ant=_log_int(rng, 60, 300),
                   n_times=rng.randint(1, 4), n_chan=rng.randint(1, 8), nside=_log_int(rng, 40, 256), **opt)
    elif kind == "ska":
        c = _ska("", eps=eps, call=call, n_ant=_log_int(rng, 100, 512), nside=_log_int(rng, 100, 700), **opt)
    elif kind == "sweep":
        r = math.exp(rng.uniform(math.log(0.3), math.log(3.0)))
        n_pix = int(130_000 * r ** 1.66)
        c = _sweep("", r, n_pix, eps=eps, call=call, ntrans=rng.choice([1, 1, 3]), **opt)
        if c["ntrans"] == 1:
            c["complex"] = rng.random() < 0.3
    elif kind == "sparse":
        c = _sweep("", math.exp(rng.uniform(math.log(1.0), math.log(10.0))), _log_int(rng, 100, 5000),
                   groups=rng.randint(1, 9), eps=eps, call=call, **opt)
    else:
        c = _ska("", eps=rng.choice([1e-4, 1e-6]), call=call, n_times=rng.randint(1, 8), uv_max=rng.uniform(250.0, 500.0),
                 nside=_log_int(rng, 128, 512), **opt)
        c["n_vis"] = _core_count(c["uv_max"], c["n_times"])
    del c["name"]
    return c


# --------------------------------------------------------------------------- geometry and values


def _ring_sizes(nside, cap_deg):
    """z and pixel count of the HEALPix RING rings with z >= cos(cap_deg) (caps up to a hemisphere)."""
    i = np.arange(1, 2 * nside + 1)
    z = np.where(i < nside, 1.0 - i * i / (3.0 * nside * nside), 4.0 / 3.0 - 2.0 * i / (3.0 * nside))
    keep = z >= math.cos(math.radians(cap_deg)) - 1e-12
    return i[keep], z[keep], np.where(i < nside, 4 * i, 4 * nside)[keep]


def _cap(nside, cap_deg, n_pix):
    """RING-ordered unit vectors of the cap (its first n_pix pixels for n_pix > 0)."""
    if nside == 0:  # the smallest resolution of a coarse ladder whose cap holds n_pix
        nside = 1
        while int(_ring_sizes(nside, cap_deg)[2].sum()) < n_pix:
            nside += max(1, nside // 8)
    ring, z, n = _ring_sizes(nside, cap_deg)
    if n_pix > 0:
        last = int(np.searchsorted(np.cumsum(n), n_pix)) + 1
        ring, z, n = ring[:last], z[:last], n[:last]
    start = np.concatenate([[0], np.cumsum(n)[:-1]])
    j = np.arange(int(n.sum())) - np.repeat(start, n)  # 0-based in its ring
    shift = np.where(ring < nside, 0.5, 1.0 - 0.5 * ((ring - nside + 1) % 2))  # in pixels of the ring
    frac = j + np.repeat(shift, n)
    phi = 2.0 * math.pi * frac / np.repeat(n, n)
    zz = np.repeat(z, n)
    st = np.sqrt(np.maximum(0.0, (1.0 - zz) * (1.0 + zz)))
    pix = np.stack([st * np.cos(phi), st * np.sin(phi), zz], axis=1)
    return pix[:n_pix] if n_pix > 0 else pix


def _antennas(c, rng):
    n, kind = c["n_ant"], c["layout"]
    if kind == "annuli":
        rings, top = [], c["r_max_m"] / 1e3
        for a, b, k in zip(_EDGES_KM[:-1], _EDGES_KM[1:], _COUNTS):  # uniform in area; the last ring in part
            if top > a:
                k = int(round(k * (min(top, b) ** 2 - a ** 2) / (b ** 2 - a ** 2)))
                rings.append(1e3 * np.sqrt(rng.uniform(a ** 2, min(top, b) ** 2, k)))
        r = np.concatenate(rings)
        n = len(r)
    elif kind == "disk":
        r = c["r_max_m"] * np.sqrt(rng.uniform(0.0, 1.0, n))
    else:
        r = np.exp(rng.uniform(math.log(c["r_min_m"]), math.log(c["r_max_m"]), n))
    t = rng.uniform(0.0, 2.0 * math.pi, n)
    ant = np.stack([r * np.cos(t), r * np.sin(t), rng.normal(0.0, c["sigma_z_m"], n)], axis=1)
    if kind == "core":  # 60 % of the antennas in a Gaussian core of 500 m
        k = int(round(0.6 * n))
        ant[:k, :2] = rng.normal(0.0, 500.0, (k, 2))
    return ant


def _baselines(c, rng):
    ant = _antennas(c, rng)
    i, j = np.triu_indices(len(ant), k=1)
    d = ant[j] - ant[i]
    lat = math.radians(c["lat"])
    axis = np.array([0.0, math.cos(lat), math.sin(lat)])
    n_times = c["n_times"]
    if c["n_vis"] > 0:
        n_times = max(n_times, -(-c["n_vis"] // len(d)))
    out = []
    for k in range(n_times):
        h = math.radians((k - (n_times - 1) / 2.0) * c["step_deg"])
        dr = d * math.cos(h) + np.cross(axis, d) * math.sin(h) + np.outer(d @ axis, axis) * (1.0 - math.cos(h))
        for lam in np.linspace(c["lam"], c["lam_max"], c["n_chan"]):
            out.append(dr / lam)
    uvw = np.concatenate(out, axis=0)
    if c["uv_max"] > 0:
        uvw = uvw[np.hypot(uvw[:, 0], uvw[:, 1]) <= c["uv_max"]]
    if c["n_vis"] > 0:
        uvw = uvw[:c["n_vis"]]
    return np.ascontiguousarray(uvw)


def _pixels(c, rng):
    if c["groups"] == 0:
        return _cap(c["nside"], c["cap_deg"], c["n_pix"])
    # compact groups of pixels of interest: square patches of the pixel pitch around drawn directions of the field
    per = -(-c["n_pix"] // c["groups"])
    side = int(math.ceil(math.sqrt(per)))
    pitch = math.sqrt(math.pi / 3.0) / c["nside"]
    gx, gy = np.meshgrid(np.arange(side) - side / 2.0, np.arange(side) - side / 2.0)
    out = []
    for _ in range(c["groups"]):
        t, f = rng.uniform(0.0, math.radians(20.0)), rng.uniform(0.0, 2.0 * math.pi)
        xy = np.stack([math.sin(t) * math.cos(f) + gx.ravel() * pitch, math.sin(t) * math.sin(f) + gy.ravel() * pitch],
                      axis=1)[:per]
        out.append(np.concatenate([xy, np.sqrt(1.0 - (xy * xy).sum(1))[:, None]], axis=1))
    return np.ascontiguousarray(np.concatenate(out)[:c["n_pix"]])


def _request(c, b):
    """Pixels, baselines and tolerance of request b of a batch: sizes log-uniform in [1e3, the case's], the first the largest."""
    if b == 0:
        return c["n_pix"], c["n_vis"], 1e-4
    rng = np.random.Generator(np.random.PCG64([c["n_pix"], c["n_vis"], b]))
    n_pix, n_vis = (int(round(math.exp(rng.uniform(math.log(1e3), math.log(c[k]))))) for k in ("n_pix", "n_vis"))
    return n_pix, n_vis, (1e-4, 1e-6, 1e-9)[b % 3]


def _jobs(c, seed):
    """The transforms of one pass: a list of (case of one transform, pixels, baselines, weights, skies, visibilities)."""
    out = []
    for b in range(c["count"]):
        rng = np.random.Generator(np.random.PCG64([int(seed), b, 20230609]))
        one = dict(c)
        if c["api"] == "batch":  # the stream's mix: log-uniform sizes up to the case's, a tolerance each
            one["n_pix"], one["n_vis"], one["eps"] = _request(c, b)
        pix, uvw = _pixels(one, rng), _baselines(one, rng)
        w = rng.uniform(0.5, 1.5, len(pix)) if c["weights"] else None
        nt = c["ntrans"]
        sky = rng.lognormal(0.0, 1.0, (nt, len(pix)))
        if c["complex"]:
            sky = sky * np.exp(2j * math.pi * rng.uniform(0.0, 1.0, sky.shape))
        vis = rng.normal(0.0, math.sqrt(0.5), (nt, len(uvw), 2)).view(np.complex128)[..., 0]
        out.append((one, pix, uvw, w, sky, vis))
    return out


def _in_precision(one, sky, vis):
    """Sky and visibilities in the precision the plan of this tolerance takes."""
    if one["eps"] >= 1e-6:
        return sky.astype(np.complex64 if np.iscomplexobj(sky) else np.float32), vis.astype(np.complex64)
    return sky, vis


# --------------------------------------------------------------------------- a pass


def prepare(case, seed):
    state = {"case": case, "plans": [], "skies": [], "vis": []}
    for one, pix, uvw, w, sky, vis in _jobs(case, seed):
        sky, vis = _in_precision(one, sky, vis)
        if case["ntrans"] == 1:
            sky, vis = sky[0], vis[0]
        if case["api"] == "noalloc":
            state["pix"], state["uvw"] = torch.as_tensor(pix, device="cuda"), torch.as_tensor(uvw, device="cuda")
            state["out"] = torch.empty(len(uvw), dtype=torch.complex64, device="cuda")
        else:
            state["plans"].append(hvox.Plan(pix, uvw, one["eps"], isign=case["isign"], weight=w, ntrans=case["ntrans"],
                                            search_threshold=case["threshold"]))
        state["skies"].append(torch.as_tensor(sky, device="cuda"))
        state["vis"].append(torch.as_tensor(vis, device="cuda"))
    return state


def run(state):
    case = state["case"]
    if case["api"] == "noalloc":
        return {"V": hvox.direct_synthesize_noalloc(state["pix"], state["uvw"], state["skies"][0], state["out"],
                                                    isign=case["isign"])}
    if case["api"] == "batch":
        if case["call"] == "predict":
            return {"V": hvox.synthesize_batch(state["plans"], state["skies"])}
        return {"I": hvox.analyze_batch(state["plans"], state["vis"])}
    plan, sky, vis = state["plans"][0], state["skies"][0], state["vis"][0]
    out = {}
    if case["call"] in ("predict", "step"):
        out["V"] = plan.synthesize_complex(sky) if case["complex"] else plan.synthesize(sky)
    if case["call"] in ("image", "step"):
        out["I"] = plan.analyze_complex(vis) if case["complex"] else plan.analyze(vis)
    return out


# --------------------------------------------------------------------------- the least work, and exact values


def _sizes(c):
    """(pixels, baselines, pixel extents, baseline extents) of one transform of the case, from geometry drawn once."""
    rng = np.random.Generator(np.random.PCG64([1, 0, 20230609]))
    pix, uvw = _pixels(c, rng), _baselines(c, rng)
    return len(pix), len(uvw), np.ptp(pix, axis=0), np.ptp(uvw, axis=0)


def work(case):
    """Inputs and outputs once each (coordinates included, as 3 FP64 a point); operations of the cheaper of the two
    evaluations: direct sums (16 a pair: a 3-term phase, one sine and cosine, a complex multiply-add) or one type-3
    transform over the whole geometry (8 a kernel tap and 5 M log2 M for its FFT) at an upsampling of 1.25."""
    total = {"bytes": 0.0, "flops": 0.0}
    if case["api"] == "batch":
        for n_pix, n_vis, eps in (_request(case, b) for b in range(case["count"])):
            size = 4 if eps >= 1e-6 else 8
            total["bytes"] += size * (n_pix + 2 * n_vis) + 24.0 * (n_pix + n_vis)
            total["flops"] += 16.0 * n_pix * n_vis
        return total
    n_pix, n_vis, P, B = _sizes(case)
    eps, sigma = case["eps"], 1.25
    size = 4 if eps >= 1e-6 else 8
    w = math.ceil(math.log(1.0 / eps) / (math.pi * math.sqrt(1.0 - 1.0 / sigma)))
    cells = 1.0
    for p, b in zip(P, B):
        cells *= max(sigma * (sigma * p * b + w + 2), 2 * w)
    nufft = 8.0 * w ** 3 * (n_pix + n_vis) + 5.0 * cells * math.log2(cells)
    calls = (2 if case["call"] == "step" else 1) * case["ntrans"] * (2 if case["complex"] else 1)
    total["bytes"] = size * (n_pix + 2 * n_vis) * calls + 24.0 * (n_pix + n_vis)
    total["flops"] = float(calls * min(16.0 * n_pix * n_vis, nufft))
    return total


_EXACT_PAIRS = 9e10  # about 20 s of FP64 sums


def exact(case, seed):
    """Direct sums in FP64. The turns <p, r> (up to ~1e5) are split so that their integer part drops without error:
    p = ph + pl with ph a multiple of 2^-8 and r = rh + rl with rh a multiple of 2^-26, so that the products and
    sums of ph rh are exact, and the rest is below 1e-2 turns."""
    jobs = _jobs(case, seed)
    if sum(len(j[1]) * len(j[2]) for j in jobs) > _EXACT_PAIRS:
        return None
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    outs = {"V": [], "I": []}
    for one, pix, uvw, w, sky, vis in jobs:
        sky, vis = (torch.as_tensor(x, device=dev).to(torch.complex128) for x in _in_precision(one, sky, vis))
        r, p = torch.as_tensor(pix, device=dev), torch.as_tensor(uvw, device=dev)
        c = sky * torch.as_tensor(w, device=dev) if w is not None else sky
        rh = torch.round(r * 2.0 ** 26) * 2.0 ** -26
        ph = torch.round(p * 2.0 ** 8) * 2.0 ** -8
        low = torch.cat([r - rh, r], dim=1).T  # (6, n_pix): ph rl + pl r
        rhT = rh.T
        cr, ci = c.real.T.contiguous(), c.imag.T.contiguous()
        V = torch.zeros(len(p), case["ntrans"], dtype=torch.complex128, device=dev)
        I = torch.zeros(len(r), case["ntrans"], dtype=torch.complex128, device=dev)
        s = float(case["isign"])
        want_v, want_i = case["call"] in ("predict", "step"), case["call"] in ("image", "step")
        rows = max(1, int(2e8 // len(r)))
        for k in range(0, len(p), rows):
            a, al = ph[k:k + rows], torch.cat([ph[k:k + rows], p[k:k + rows] - ph[k:k + rows]], dim=1)
            t = (a @ rhT).frac_().addmm_(al, low).mul_(2.0 * math.pi)
            sn = torch.sin(t)
            cs = t.cos_()
            if want_v:  # V = sum c e^{s j t}
                re, im = cs @ cr, s * (sn @ cr)
                if case["complex"]:
                    re, im = re - s * (sn @ ci), im + cs @ ci
                V[k:k + rows] = torch.complex(re, im)
            if want_i:  # I = w sum V e^{-s j t}
                vr, vi = (x.T.contiguous() for x in (vis[:, k:k + rows].real, vis[:, k:k + rows].imag))
                re = cs.T @ vr + s * (sn.T @ vi)
                im = cs.T @ vi - s * (sn.T @ vr) if case["complex"] else torch.zeros_like(re)
                I += torch.complex(re, im)
            del t, sn, cs
        if w is not None:
            I = I * torch.as_tensor(w, device=dev)[:, None]
        if not case["complex"]:
            I = I.real
        V, I = V.T.contiguous(), I.T.contiguous()
        if case["ntrans"] == 1:
            V, I = V[0], I[0]
        if want_v:
            outs["V"].append(V)
        if want_i:
            outs["I"].append(I)
    batch = case["api"] == "batch"
    return {k: (v if batch else v[0]) for k, v in outs.items() if v}
