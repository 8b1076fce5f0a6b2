"""The work that programs have this library do, as cases to be timed: photon
propagation of showers (device, batched and host calls; plane and spherical
shell; tables, stepper and network; Cherenkov and fluorescence light; with and
without mirrors) and the training and evaluation of the learned correction.

A case is a dict of plain values; ``listed()`` names the usual ones, ``draw``
gives others of the same ranges, ``prepare`` makes what a program holds before
the call (segments in device or pinned memory, atmosphere, detector, network,
output buffers), ``run`` is one call through the library's entry points.
``exact`` follows the plain method in 64 bits for the plane's Cherenkov light.
"""
from __future__ import annotations

import ctypes as C
import math

import numpy as np
import torch

from paper_2405_04229_gb300 import binding as B
from paper_2405_04229_gb300 import synth

C_LIGHT = 299_792_458.0
H_OBS = 2000.0
LAMBDA_NM = (300.0, 600.0)
ALPHA = 7.2973525693e-3

PROPAGATE = dict(path="device", geometry="planar", segments=0, showers=1, uneven=False, zenith=20.0, energy=1e12,
                 bunch=5, refraction=True, transmission=True, telescopes=100, emission="cherenkov", tracer="tables",
                 optics=False, surrogate=False, lv3=False)


def _case(name, **kw):
    return dict(PROPAGATE, name=name, **kw)


def listed():
    return [
        # the smallest use: a thousand tracks in straight lines, every photon by itself, no array
        _case("tiny_straight", segments=1000, zenith=0.0, energy=1e12, bunch=1, refraction=False, transmission=False,
              telescopes=0),
        # one small event handed over by a shower program, every photon by itself, 100 telescopes
        _case("single_event", segments=5003, bunch=1),
        # the ordinary refraction-corrected batch: 10 showers of 1e5 segments
        _case("showers_planar", segments=1_000_000, showers=10),
        # many showers of uneven size and bunch size in one captured launch, 400 telescopes
        _case("batch_uneven", path="batch", segments=4_000_037, showers=24, uneven=True, zenith=40.0, bunch=0,
              telescopes=400),
        # a chunk of a large inclined shower through the spherical shell, 2,000 telescopes
        _case("inclined_sphere", geometry="spherical", segments=10_000_000, zenith=60.0, energy=1e14, bunch=10,
              telescopes=2000),
        # nitrogen fluorescence of the same showers: a quarter of it beyond the tables
        _case("fluorescence_half", segments=1_000_000, showers=10, emission="fluorescence_half"),
        # mirrors and cameras behind every telescope sphere
        _case("optics_camera", segments=1_000_000, showers=10, optics=True),
        # the learned correction in the place of the tables
        _case("surrogate_planar", segments=1_000_000, showers=10, surrogate=True),
        # the per-photon Snell stepper, the tracer for any atmosphere
        _case("snell_planar", segments=100_000, showers=10, tracer="snell"),
        # segments and outputs in the host's pinned memory, as a shower program on the host has them
        _case("host_call", path="host", segments=1_000_000, showers=10),
        # training the learned correction (shortened: 320 of 51,200 Adam steps)
        dict(name="surrogate_train", path="train", samples=262_144, batch=32_768, epochs=40, split=False),
        # the learned correction by itself over a list of points
        dict(name="surrogate_eval", path="eval", points=1_000_003, split=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["straight", "device", "device", "batch", "spherical", "spherical", "fluorescence", "optics",
                       "surrogate", "snell", "host", "train", "eval"])
    zen = round(rng.uniform(0.0, 40.0), 2)
    n_showers = rng.randint(1, 12)
    if kind == "straight":
        return dict(PROPAGATE, segments=_log_int(rng, 200, 500_000), zenith=zen, bunch=rng.choice([1, 2, 5]),
                    refraction=False, transmission=rng.random() < 0.5, telescopes=rng.choice([0, 100]))
    if kind == "device":
        return dict(PROPAGATE, segments=_log_int(rng, 1000, 3_000_000), showers=n_showers, zenith=zen,
                    bunch=rng.choice([2, 3, 5, 10]), telescopes=rng.choice([100, 400]), lv3=rng.random() < 0.25)
    if kind == "batch":
        return dict(PROPAGATE, path="batch", segments=_log_int(rng, 100_000, 6_000_000), showers=rng.randint(4, 48),
                    uneven=True, zenith=40.0, bunch=0, telescopes=rng.choice([100, 400]))
    if kind == "spherical":
        return dict(PROPAGATE, geometry="spherical", segments=_log_int(rng, 10_000, 8_000_000),
                    zenith=round(rng.uniform(20.0, 65.0), 2), energy=1e14, bunch=rng.choice([5, 10]),
                    telescopes=rng.choice([100, 2000]), lv3=rng.random() < 0.25)
    if kind == "fluorescence":
        return dict(PROPAGATE, segments=_log_int(rng, 10_000, 2_000_000), showers=n_showers, zenith=zen,
                    geometry=rng.choice(["planar", "planar", "spherical"]), bunch=rng.choice([1, 5]),
                    emission=rng.choice(["fluorescence", "fluorescence_half"]))
    if kind == "optics":
        return dict(PROPAGATE, segments=_log_int(rng, 10_000, 1_500_000), showers=n_showers, zenith=zen, optics=True)
    if kind == "surrogate":
        return dict(PROPAGATE, segments=_log_int(rng, 5_000, 1_200_000), showers=n_showers, zenith=zen, surrogate=True)
    if kind == "snell":
        return dict(PROPAGATE, segments=_log_int(rng, 1_000, 150_000), showers=n_showers, zenith=zen, tracer="snell",
                    geometry=rng.choice(["planar", "planar", "spherical"]))
    if kind == "host":
        return dict(PROPAGATE, path="host", segments=_log_int(rng, 1_000, 2_000_000), showers=n_showers, zenith=zen,
                    bunch=rng.choice([2, 5]))
    if kind == "train":
        batch = rng.choice([4096, 16_384, 32_768])
        return dict(path="train", samples=batch * rng.randint(2, 8) + rng.choice([0, 0, 17]), batch=batch,
                    epochs=rng.randint(5, 40), split=rng.random() < 0.3)
    return dict(path="eval", points=_log_int(rng, 100, 4_000_000), split=rng.random() < 0.3)


# --- inputs ---------------------------------------------------------------------------------------


def _generator(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed((seed * 1_000_003 + stream) & 0x7FFFFFFF)
    return g


def _greisen_quantiles(E0_eV, X_cut, Ec_eV=81e6, X0=36.7):
    """(CDF, slant depth) of the Greisen profile truncated at X_cut, 20,001 nodes."""
    beta0 = math.log(E0_eV / Ec_eV)
    t = np.linspace(1e-4, X_cut / X0, 20001)
    s = 3.0 * t / (t + 2.0 * beta0)
    dens = np.exp(t * (1.0 - 1.5 * np.log(s)))
    cdf = np.concatenate([[0.0], np.cumsum(0.5 * (dens[1:] + dens[:-1]) * np.diff(t))])
    return cdf / cdf[-1], t * X0


def _heights(X):
    """Heights of vertical column depths X [g/cm^2] in the standard atmosphere."""
    p = synth.US_STANDARD
    h = torch.zeros_like(X)
    for i in range(5):
        lo = p["layer_h"][i]
        if i < 4:
            hi = -torch.log(((X - p["a"][i]) / p["b"][i]).clamp_min(1e-300)) * p["c"][i] / 100.0
        else:
            hi = (p["a"][i] - X) * p["c"][i] / p["b"][i] / 100.0
        h = torch.where(hi >= lo, hi, h) if i else hi
    return h


def _shower(n, zenith_deg, azimuth_deg, E0_eV, gen, shower_id):
    """n segments of a synthetic shower (the profile and spreads of the package's
    own synthetic showers) as an (n, 64) byte tensor on the device."""
    dev = gen.device
    f64 = dict(dtype=torch.float64, device=dev)
    th, ph = math.radians(zenith_deg), math.radians(azimuth_deg)
    back = torch.tensor([math.sin(th) * math.cos(ph), math.sin(th) * math.sin(ph), math.cos(th)], **f64)
    e1 = torch.tensor([-math.sin(ph), math.cos(ph), 0.0], **f64)
    e2 = torch.linalg.cross(-back, e1)
    X_ground = float(synth._column_depth(np.array([H_OBS]))[0])
    cdf, depth = (torch.from_numpy(a).to(dev) for a in _greisen_quantiles(E0_eV, X_ground / math.cos(th)))
    u = torch.rand(n, generator=gen, **f64)
    j = torch.searchsorted(cdf, u).clamp(1, len(cdf) - 1)
    X = depth[j - 1] + (u - cdf[j - 1]) / (cdf[j] - cdf[j - 1]).clamp_min(1e-300) * (depth[j] - depth[j - 1])
    h = _heights((X * math.cos(th)).clamp_max(X_ground))
    lat = 20.0 * torch.randn(n, 2, generator=gen, **f64)
    pos = ((h - H_OBS) / math.cos(th))[:, None] * back + lat[:, :1] * e1 + lat[:, 1:] * e2
    pos[:, 2] += H_OBS
    ang = torch.tan(math.radians(3.0) * torch.randn(n, 2, generator=gen, **f64))
    d = -back + ang[:, :1] * e1 + ang[:, 1:] * e2
    d /= d.norm(dim=1, keepdim=True)
    seg = torch.zeros(n, 8, **f64)
    seg[:, :3] = pos
    seg[:, 3] = (synth.US_STANDARD["h_top"] - h) / math.cos(th) / C_LIGHT
    f = seg.view(torch.float32)
    f[:, 8:11] = d.float()
    f[:, 11] = 1.0 + 4.0 * torch.rand(n, generator=gen, dtype=torch.float32, device=dev)
    gamma = torch.exp(math.log(50.0) + math.log(200.0) * torch.rand(n, generator=gen, **f64))
    f[:, 12] = (1.0 / gamma**2).float()
    f[:, 13] = (2 * torch.randint(0, 2, (n,), generator=gen, device=dev) - 1).float()
    seg.view(torch.int32)[:, 14] = shower_id
    return seg.view(torch.uint8).reshape(n, 64)


def _segments(case, seed):
    """The case's showers one after the other, and the number of segments of each."""
    rng = np.random.default_rng([seed, 0x5E6])
    n, k = case["segments"], case["showers"]
    if case["uneven"]:   # log-uniform over two decades, zenith and azimuth of each shower its own
        share = 10.0 ** rng.uniform(0.0, 2.0, k)
        counts = np.maximum(1, np.floor(share / share.sum() * n)).astype(np.int64)
        zen, azi = rng.uniform(0.0, case["zenith"], k), rng.uniform(0.0, 360.0, k)
    else:
        counts = np.full(k, n // k, np.int64)
        zen, azi = np.full(k, case["zenith"]), np.zeros(k)
    counts[-1] += n - counts.sum()
    parts = [_shower(int(c), zen[i], azi[i], case["energy"], _generator(seed, i), i) for i, c in enumerate(counts)]
    return torch.cat(parts), counts


def _telescopes(n):
    if n == 2000:
        return synth.poisson_disk_telescopes(n=2000, half=1000.0, min_sep=13.0, radius=6.0, seed=0)
    side = int(round(math.sqrt(n)))
    return synth.grid_telescopes(nx=side, ny=side, pitch=100.0) if n else None


class _Batch:
    """Owns a cs_batch handle."""

    def __init__(self, handle):
        self.handle = handle

    def __del__(self):
        B.cs_batch_destroy(self.handle)


def _train(atm, seed, samples, batch, epochs, split):
    return B.Surrogate(atm, n_train=samples, n_heldout=16_384, batch=batch, epochs=epochs, seed=seed,
                       split_activations=int(split))


def _options(case, state):
    o = B.cs_opts_default()
    o.bunch, o.device_ptrs = max(case["bunch"], 1), int(case["path"] != "host")
    if case["tracer"] == "snell":
        o.tracer, o.tracer_dh = B.CS_TRACER_SNELL, 10.0
    if case["emission"] != "cherenkov":
        state["lines"] = B.set_fluorescence(o, dict(synth.FLUORESCENCE, half=case["emission"] == "fluorescence_half"))
    if case["lv3"]:   # a disc that holds the array and its histogram, and 60 m for the correction
        B.set_lv3(o, dict(centre=(0.0, 0.0, H_OBS), radius=1420.0 if case["telescopes"] >= 400 else 700.0, margin=60.0))
    if case["surrogate"]:
        o.surrogate = state["surrogate"].handle
    return o


def prepare(case, seed):
    st = {"case": case, "seed": seed}
    if case["path"] in ("train", "eval"):
        st["atm"] = B.Atmosphere(layered=synth.US_STANDARD, refraction=True, transmission=True)
        if case["path"] == "eval":
            st["surrogate"] = _train(st["atm"], seed, 65_536, 32_768, 4, case["split"])
            g = _generator(seed, 77)
            u = torch.rand(case["points"], 3, generator=g, device="cuda")
            x = torch.zeros(case["points"], 4, device="cuda")
            x[:, 0] = 28_000.0 * u[:, 0]                             # emission height above the array [m]
            x[:, 1] = torch.cos(math.radians(60.0) * u[:, 1])        # cosine of the zenith
            x[:, 2] = 1.0 / (300.0 + 300.0 * u[:, 2])                # 1 / wavelength [1/nm]
            st["in"], st["out"] = x, torch.empty_like(x)
        return st
    sph = case["geometry"] == "spherical"
    st["atm"] = B.Atmosphere(layered=synth.US_STANDARD, refraction=case["refraction"],
                             transmission=case["transmission"], spherical=sph)
    optics = dict(mirror_d=7.0, focal_f=8.0, camera_r=0.5, point_zenith=math.radians(case["zenith"]),
                  point_azimuth=0.0, cam_n=41) if case["optics"] else None
    st["det"] = det = B.Detector(n_showers=case["showers"], hist=synth.histogram_400(),
                                 tel=_telescopes(case["telescopes"]), spherical=sph, optics=optics)
    if case["surrogate"]:
        st["surrogate"] = _train(st["atm"], seed, 65_536, 32_768, 4, False)
    segs, counts = _segments(case, seed)
    st["opts"] = _options(case, st)
    if case["path"] == "host":
        st["segs"] = segs.cpu().pin_memory()
        pinned = dict(pin_memory=True, dtype=torch.int64)
        st["hist"] = torch.zeros(det.n_showers, 400, 400, **pinned)
        st["tel_counts"] = torch.zeros(det.n_showers, det.n_tel, **pinned)
        st["tel_time"] = torch.zeros(det.n_showers, det.n_tel, dtype=torch.float64, pin_memory=True)
        st["counters"] = torch.zeros(B.CS_N_COUNTERS, **pinned)
        o = st["out"] = B.cs_output()
        o.hist, o.tel_counts = st["hist"].data_ptr(), st["tel_counts"].data_ptr()
        o.tel_time, o.counters = st["tel_time"].data_ptr(), st["counters"].data_ptr()
        return st
    st["segs"], st["outs"] = segs, B.DeviceOutputs(det)
    if case["path"] == "batch":   # bunch sizes as the autotuner picks them: larger for the larger showers
        order = np.argsort(np.argsort(counts))
        bunches = np.array([1, 2, 5, 10], np.int32)[order * 4 // len(counts)]
        st["bunches"] = bunches
        st["batch"] = _Batch(B.cs_batch_create(C.c_void_p(segs.data_ptr()), len(segs), st["atm"].handle, det.handle,
                                               seed, bunches, st["opts"], st["outs"].out))
    return st


def run(state):
    case, path = state["case"], state["case"]["path"]
    if path == "train":
        sur = _train(state["atm"], state["seed"], case["samples"], case["batch"], case["epochs"], case["split"])
        params, norm = sur.info()
        return {"params": params, "norm": norm, "loss": sur.stats["final_loss"], "heldout_p99": np.array(sur.stats["p99"])}
    if path == "eval":
        st = B.lib().cs_surrogate_eval(state["surrogate"].handle, C.c_void_p(state["in"].data_ptr()), case["points"],
                                       C.c_void_p(state["out"].data_ptr()), B.stream_ptr())
        if st != B.CS_OK:
            raise B.CSError(st, "cs_surrogate_eval")
        return {"fields": state["out"]}
    if path == "batch":
        st = B.cs_batch_launch(state["batch"].handle, B.stream_ptr())
    else:
        out = state["out"] if path == "host" else state["outs"].out
        st = B.cs_propagate_ex(C.c_void_p(state["segs"].data_ptr()), case["segments"], state["atm"].handle,
                               state["det"].handle, state["seed"], state["opts"], out, B.stream_ptr())
    if st != B.CS_OK:
        raise B.CSError(st, "cs_propagate_ex")
    o = state if path == "host" else vars(state["outs"])
    res = {"hist": o["hist"], "counters": o["counters"]}
    if case["telescopes"]:
        res["tel_counts"], res["tel_time"] = o["tel_counts"], o["tel_time"]
    if case["optics"]:
        res["camera"] = o["camera"]
    return res


def work(case):
    if case["path"] == "train":
        steps = case["samples"] // case["batch"] * case["epochs"]
        macs = 3 * 64 + 2 * 64 * 64 + 3 * 64
        return {"bytes": steps * case["batch"] * 9 * 4, "flops": 6 * macs * steps * case["batch"]}
    if case["path"] == "eval":
        return {"bytes": case["points"] * 32, "flops": case["points"] * 2 * (3 * 64 + 2 * 64 * 64 + 3 * 64)}
    n = case["segments"]
    outputs = case["showers"] * (400 * 400 + 2 * case["telescopes"] + (41 * 41 * case["telescopes"] if case["optics"] else 0))
    # per segment 3 m of track in 3.5 sub-steps; about 16 photons a metre (fluorescence: 1.6).  Lane
    # operations of the method's formulas per segment, per sub-step and per bunch.
    per_metre = 16.0 if case["emission"] == "cherenkov" else 1.6
    bunches = n * 3.0 * per_metre / (case["bunch"] or 4)
    per_bunch = 285.0 + (85.0 if case["geometry"] == "spherical" else 0.0)
    if case["tracer"] == "snell":
        per_bunch += 800 * 30.0
    if case["surrogate"]:
        per_bunch += 2 * (3 * 64 + 2 * 64 * 64 + 3 * 64)
    return {"bytes": 64 * n + 8 * outputs, "flops": 120.0 * n + 150.0 * 3.5 * n + per_bunch * bunches}


# --- the plain method in 64 bits ------------------------------------------------------------------


def _mulhi(a, c):
    return ((a * (c >> 16)) + ((a * (c & 0xFFFF)) >> 16)) >> 16


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 (Salmon et al. 2011) on int64 tensors holding 32-bit words."""
    M = 0xFFFFFFFF
    k0, k1 = seed & M, (seed >> 32) & M
    for _ in range(10):
        h0, l0 = _mulhi(0xD2511F53, c0), (0xD2511F53 * c0) & M
        h1, l1 = _mulhi(0xCD9E8D57, c2), (0xCD9E8D57 * c2) & M
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
    return [(c >> 8).double() * 2.0**-24 for c in (c0, c1, c2, c3)]


def _density(h):
    """Density [g/cm^3] of the standard atmosphere at heights h [m]."""
    p = synth.US_STANDARD
    rho = torch.zeros_like(h)
    for i in range(5):
        c = p["c"][i]
        law = p["b"][i] / c * (torch.exp(-100.0 * h / c) if i < 4 else torch.ones_like(h))
        rho = torch.where(h >= p["layer_h"][i], law, rho) if i else law
    return torch.where(h < p["h_top"], rho, torch.zeros_like(rho))


def _delta(h):
    return synth.US_STANDARD["kappa"] * _density(h) / (synth.US_STANDARD["b"][0] / synth.US_STANDARD["c"][0])


def _optical_depth(X, A, inv_l):
    """Rayleigh and aerosol optical depth of slant columns X [g/cm^2], A [m] at 1 / inv_l [nm]."""
    t = synth.TRANSMISSION
    return (X / t["rayl_X0"] * (t["rayl_lambda0"] * 1e9 * inv_l) ** 4
            + t["aer_tau0"] * (t["aer_lambda0"] * 1e9 * inv_l) ** t["aer_alpha"] * A / t["aer_H"])


_EDGES = [H_OBS, 4000.0, 7000.0, 10000.0, 20000.0, 40000.0, 70000.0, 100000.0, 112829.2]


def _refracted(he, cos0):
    """Displacement over sin(zenith), c x optical time, slant density and aerosol columns of the
    planar path with n sin(theta) conserved (Gauss-Legendre over the layers)."""
    x, w = (torch.from_numpy(v).to(he.device) for v in np.polynomial.legendre.leggauss(16))
    ne, s2 = 1.0 + _delta(he), 1.0 - cos0**2
    D = torch.zeros_like(he)
    cT, X, A = D.clone(), D.clone(), D.clone()
    for lo, hi in zip(_EDGES[:-1], _EDGES[1:]):
        if not bool((he > lo).any()):
            break
        half = 0.5 * (he.clamp(lo, hi) - lo)
        h = lo + half[:, None] * (1.0 + x)
        wt = half[:, None] * w
        rho = _density(h)
        n = 1.0 + _delta(h)
        q = torch.sqrt((n**2 - (ne**2 * s2)[:, None]).clamp_min(1e-30))
        D += (wt * ne[:, None] / q).sum(1)
        cT += (wt * n**2 / q).sum(1)
        X += (wt * 100.0 * rho * n / q).sum(1)
        A += (wt * torch.exp(-h / synth.TRANSMISSION["aer_H"]) * n / q).sum(1)
    return D, cT, X, A


def _exact_times(case, seed, segs, counts, bunches):
    """Per shower and telescope, the sum over hits of bunch size x arrival time [s]."""
    tel = torch.from_numpy(_telescopes(case["telescopes"])).cuda()
    out = torch.zeros(case["showers"] * len(tel), dtype=torch.float64, device="cuda")
    size = torch.as_tensor(bunches, device="cuda").double()
    il = [1.0 / v for v in LAMBDA_NM]
    frank_tamm = 2.0 * math.pi * ALPHA * (il[0] - il[1]) * 1e9
    n_obs = 1.0 + float(_delta(torch.tensor([H_OBS], dtype=torch.float64))[0])
    step = max(500, 20_000_000 // (len(tel) * 12))
    for first in range(0, len(segs), step):
        raw = segs[first:first + step]
        d, f, i32 = raw.view(torch.float64), raw.view(torch.float32).double(), raw.view(torch.int32)
        gid = torch.arange(first, first + len(raw), device="cuda")
        P = f[:, 8:11] / f[:, 8:11].norm(dim=1, keepdim=True)
        L, g, z2, sh = f[:, 11], f[:, 12], f[:, 13] ** 2, i32[:, 14].long()
        # sub-steps of at most 1 m: angle and mean bunch count at the midpoint
        K = torch.ceil(L).long().clamp_min(1)
        s = torch.repeat_interleave(torch.arange(len(raw), device="cuda"), K)
        k = torch.arange(len(s), device="cuda") - torch.repeat_interleave(K.cumsum(0) - K, K)
        dl = (L / K)[s]
        dm = _delta(d[s, 2] + (k + 0.5) * dl * P[s, 2])
        sin2 = 1.0 - 1.0 / ((1.0 - g[s]) * (1.0 + dm) ** 2)
        mean = frank_tamm * z2[s] * sin2.clamp_min(0.0) * dl / size[sh[s]]
        u = _philox(gid[s], torch.zeros_like(s), k, torch.full_like(s, 0xFFFFFFFF), seed)[0]
        N = (mean.floor() + (u < mean - mean.floor())).long()
        # bunches: emission point, direction on the cone, wavelength
        q = torch.repeat_interleave(torch.arange(len(s), device="cuda"), N)
        i = torch.arange(len(q), device="cuda") - torch.repeat_interleave(N.cumsum(0) - N, N)
        s, k, dl, dm, sin2 = s[q], k[q], dl[q], dm[q], sin2[q]
        u0, u1, u2, u3 = _philox(gid[s], torch.zeros_like(s), k, i, seed)
        ell = (k + u0) * dl
        p, E = P[s], d[s, :3] + ell[:, None] * P[s]
        c, sn = torch.cos(2.0 * math.pi * u1), torch.sin(2.0 * math.pi * u1)
        ce = (p[:, 0] * c + p[:, 1] * sn) / (1.0 - p[:, 2])
        m = torch.stack([p[:, 0] * ce - c, p[:, 1] * ce - sn, (p[:, 2] - 1.0) * ce], 1)
        v = (1.0 - sin2).sqrt()[:, None] * p + sin2.sqrt()[:, None] * m
        inv_l = il[0] - u2 * (il[0] - il[1])
        keep = (v[:, 2] < 0.0) & (E[:, 2] >= H_OBS)
        s, dm, ell, E, v, inv_l, u3 = (t[keep] for t in (s, dm, ell, E, v, inv_l, u3))
        cos0 = -v[:, 2]
        if case["refraction"]:
            D, cT, X, A = _refracted(E[:, 2], cos0)
            ground, scale = E[:, :2] + D[:, None] * v[:, :2], (1.0 + dm) / n_obs
        else:
            dz = E[:, 2] - H_OBS
            ground, cT, scale = E[:, :2] + (dz / cos0)[:, None] * v[:, :2], dz / cos0, torch.ones_like(dm)
            zero = torch.ones_like(cos0)
            X, A = (_refracted(E[:, 2], zero)[j] / cos0 for j in (2, 3)) if case["transmission"] else (0.0, 0.0)
        if case["transmission"]:
            live = u3 < torch.exp(-_optical_depth(X, A, inv_l))
            s, ell, v, ground, scale, cT = (t[live] for t in (s, ell, v, ground, scale, cT))
        # the sphere whose centre lies closest to the arrival line
        a = v[:, :2] * scale[:, None]
        a = torch.cat([a, -torch.sqrt(1.0 - (a**2).sum(1, keepdim=True))], 1)
        near = (ground.abs() < 1000.0 + 100.0).all(1)
        s, ell, a, ground, cT = (t[near] for t in (s, ell, a, ground, cT))
        to = torch.cat([tel[None, :, :2] - ground[:, None], (tel[:, 2] - H_OBS)[None, :, None].expand(len(s), -1, 1)], 2)
        d2 = (to**2).sum(2) - (to * a[:, None]).sum(2) ** 2
        d2 = torch.where(d2 < tel[:, 3] ** 2, d2, torch.inf)
        best, which = d2.min(1)
        hit = torch.isfinite(best)
        time = d[s, 3] + ell / (torch.sqrt(1.0 - g[s]) * C_LIGHT) + cT / C_LIGHT
        slot = sh[s] * len(tel) + which
        out.index_add_(0, slot[hit], (size[sh[s]] * time)[hit])
    return out.reshape(case["showers"], len(tel))


def _exact_fields(case, seed):
    """The trained network (its own weights) and the first-order baseline, evaluated in 64 bits."""
    st = prepare(case, seed)
    p, norm = st["surrogate"].info()
    p, norm = torch.from_numpy(B.mlp_padded_to_flat(p)).double().cuda(), norm.astype(np.float64)
    x = st["in"].double()
    dz, mu, inv_l = x[:, 0], x[:, 1], x[:, 2]
    v = torch.stack([torch.exp(-dz / 8000.0), mu, inv_l], 1)
    a = v * torch.from_numpy(norm[0:3]).cuda() + torch.from_numpy(norm[3:6]).cuda()
    at = 0
    for n_in, n_out in ((3, 64), (64, 64), (64, 64), (64, 3)):
        W, b = p[at:at + n_in * n_out].reshape(n_out, n_in), p[at + n_in * n_out:at + (n_in + 1) * n_out]
        a = a @ W.T + b
        a = torch.tanh(a) if n_out == 64 else a
        at += (n_in + 1) * n_out
    y = a * torch.from_numpy(norm[6:9]).cuda() + torch.from_numpy(norm[9:12]).cuda()
    # vertical integrals of n - 1, the density and the aerosol profile from the array up
    he = H_OBS + dz
    one = torch.ones_like(he)
    _, _, X, A = _refracted(he, one)
    par = synth.US_STANDARD
    Xv = torch.zeros_like(he)
    for i in range(5):
        lo = max(par["layer_h"][i], H_OBS)
        hi = he.clamp(lo, par["layer_h"][i + 1]) if i < 4 else he.clamp_min(lo)
        c = par["c"][i] / 100.0
        Xv += par["b"][i] * (math.exp(-lo / c) - torch.exp(-hi / c)) if i < 4 else par["b"][i] * (hi - lo) / c
    rho0 = par["b"][0] / par["c"][0]
    I, de = par["kappa"] * Xv / (100.0 * rho0), _delta(he)
    Av = synth.TRANSMISSION["aer_H"] * (math.exp(-H_OBS / synth.TRANSMISSION["aer_H"]) - torch.exp(-he / synth.TRANSMISSION["aer_H"]))
    base = torch.stack([de * dz - I, 2.0 * I - de * dz + (de * dz - I) / mu**2, -_optical_depth(Xv, Av, inv_l) / mu], 1)
    f = y + base
    out = torch.zeros_like(x)
    out[:, :2] = f[:, :2]
    out[:, 2] = torch.exp(f[:, 2]).clamp_max(1.0)
    return out


def exact(case, seed):
    if case["path"] == "train":
        return None   # hundreds of steps, each on weights rounded to 16 bits: no 64-bit value to compare with
    if case["path"] == "eval":
        return {"fields": _exact_fields(case, seed)}
    res = {"hist": None, "counters": None}   # photon counts: whole numbers
    if case["optics"]:
        res["camera"] = None
    if case["telescopes"]:
        res["tel_counts"] = res["tel_time"] = None
        # the plane's Cherenkov light; the shell, the stepper, the network and light beyond the tables
        # would need a path integral of thousands of steps per photon
        plain = case["geometry"] == "planar" and case["emission"] == "cherenkov" and case["tracer"] == "tables" \
            and not case["surrogate"] and not case["lv3"] and case["segments"] * max(1, case["telescopes"] // 100) <= 1_500_000
        if plain:
            segs, counts = _segments(case, seed)
            bunches = [case["bunch"]] * case["showers"]
            if case["path"] == "batch":
                order = np.argsort(np.argsort(counts))
                bunches = np.array([1, 2, 5, 10])[order * 4 // len(counts)]
            res["tel_time"] = _exact_times(case, seed, segs, counts, bunches)
    return res if any(v is not None for v in res.values()) else None
