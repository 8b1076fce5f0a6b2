"""Telescope hits on the borders of the search's lists.  A photon's spheres are
taken from one of nine lists by its arrival zenith, or from all of them beyond
the last; each list holds the cells that its own largest zenith can reach.
Photons aimed at every sphere's disc and a little beyond its rim, from zeniths
on both sides of each border, hit what the oracle's search over all spheres
hits: spheres on the observation level, 100 m above and 100 m below it, about
the frame's origin and 39 km away (where the sphere's vertical leans 0.35 deg)."""
import math

import numpy as np
import pytest

import oracle
from paper_2405_04229_gb300 import binding as B
from paper_2405_04229_gb300 import synth
from tests import parity_util as PU

BORDERS = (24.0, 34.0, 45.0, 60.0, 67.0, 75.0, 77.0, 79.0, 82.0)   # list zeniths [deg], detector.cu
RADIUS = 6.0
H_OBS = 2000.0
ORC_ATM = oracle.make_atm(oracle.ATM_LAYERED, layered=synth.US_STANDARD)
# as in the other tests of the sphere: a few ulps of FP32 ground points tens of km away
BANDS = dict(band_pos=0.03)
FAR = (30000.0, -25000.0)


def spheres(centre, n=45):
    rng = np.random.default_rng(45)
    t = np.empty((n, 4))
    t[:, :2] = np.asarray(centre) + rng.uniform(-300.0, 300.0, (n, 2))
    t[:, 2] = H_OBS + 100.0 * (np.arange(n) % 3 - 1.0)
    t[:, 3] = RADIUS
    return t


def aimed_segments(tel, per_border, seed, spherical):
    """Tracks whose line passes within 1.3 radii of a sphere's centre, 1.5 deg to both sides of
    each border in the frame, started 30 .. 300 m above the ground."""
    rng = np.random.default_rng([seed, 0xB0])
    n = per_border * len(BORDERS)
    th = np.radians(np.repeat(BORDERS, per_border) + rng.uniform(-1.5, 1.5, n))
    ph, rot = rng.uniform(0.0, 2.0 * math.pi, (2, n))
    d = np.stack([np.sin(th) * np.cos(ph), np.sin(th) * np.sin(ph), -np.cos(th)], axis=1)
    e1 = np.stack([np.sin(ph), -np.cos(ph), np.zeros(n)], axis=1)
    e2 = np.cross(d, e1)
    off = 1.3 * RADIUS * np.sqrt(rng.uniform(0.0, 1.0, n))
    which = rng.integers(0, len(tel), n)
    centre = tel[which, :3].copy()
    ground_z = np.full(n, H_OBS)
    if spherical:
        centre = np.array([oracle.ae_inverse(t[0], t[1], t[2] - H_OBS) for t in tel])[which]
        ground_z = np.array([oracle.ae_inverse(t[0], t[1], 0.0)[2] for t in tel])[which]
    p = centre + off[:, None] * (np.cos(rot)[:, None] * e1 + np.sin(rot)[:, None] * e2)
    start_z = ground_z + rng.uniform(30.0, 300.0, n)
    p += d * ((start_z - p[:, 2]) / d[:, 2])[:, None]
    s = synth._empty(n)
    s["x0"], s["y0"], s["z0"] = p.T
    s["ux"], s["uy"], s["uz"] = d.T.astype(np.float32)
    s["length"][:] = 2.0
    s["inv_gamma2"][:] = np.float32(1e-8)
    return s


def run_oracle(segs, tel, refr, spherical):
    return oracle.propagate(segs, ORC_ATM, tel=tel, bunch=1, refraction=refr, transmission=refr, seed=3,
                            spherical=spherical, bands=BANDS)


def reach(tel, theta):
    return tel[:, 3] / math.cos(theta) + np.abs(tel[:, 2] - H_OBS) * math.tan(theta)


def test_photons_use_the_last_degree_of_every_list():
    """The inputs ask for what is tested: at every border the oracle's hits include ones below it
    whose ground point a list made for one degree less would not reach, and ones above it."""
    tel = spheres((0.0, 0.0))
    o = run_oracle(aimed_segments(tel, 300, 1, False), tel, False, False)["records"]
    o = o[(o["status"] == oracle.ST_LANDED) & (o["tel"] >= 0)]
    zen = np.degrees(np.arccos(-o["uz"]))
    gap = np.hypot(o["x"] - tel[o["tel"], 0], o["y"] - tel[o["tel"], 1])
    for b in BORDERS:
        below = (zen > b - 1.0) & (zen <= b)
        assert np.sum(below & (gap > reach(tel, math.radians(b - 1.0))[o["tel"]])) > 0, b
        assert np.sum((zen > b) & (zen < b + 1.0)) > 500, b


@pytest.mark.gpu
@pytest.mark.parametrize("centre", [(0.0, 0.0), FAR])
@pytest.mark.parametrize("spherical", [False, True])
@pytest.mark.parametrize("refr", [False, True])
def test_hits_on_the_borders_match_the_oracle(centre, spherical, refr):
    import __graft_entry__
    __graft_entry__.build()
    tel = spheres(centre)
    segs = aimed_segments(tel, 300, 2, spherical)
    atm = B.Atmosphere(layered=synth.US_STANDARD, refraction=refr, transmission=refr, spherical=spherical)
    det = B.Detector(tel=tel, spherical=spherical)
    g = B.propagate_host(segs, atm, det, seed=3, bunch=1, records=True)
    o = run_oracle(segs, tel, refr, spherical)
    st = PU.compare(g, o, bunch=1)
    assert st["matched"] > 50000 and int(g["counters"][B.CS_CNT_TEL]) > 15000
    PU.check_conservation(g["counters"])
    # without records, as a launch of one round and as a larger one
    for many, per_sm in ((segs, 0), (aimed_segments(tel, 3000, 4, spherical), 1)):
        r, c = (B.propagate_host(many, atm, det, seed=3, bunch=1, records=rec, blocks_per_sm=per_sm) for rec in (True, False))
        assert np.array_equal(c["tel_counts"], r["tel_counts"]) and np.array_equal(c["counters"], r["counters"])
