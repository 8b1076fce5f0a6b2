"""The steppers' kept layer against the general n(h) at the layer boundaries:
photons emitted at, just above and just below each boundary and above the top,
with slabs that end on, before and after it, against the FP64 oracle."""
import numpy as np
import pytest

import oracle
from tests import parity_util as PU

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dh", [7.0, 250.0, 1999.0])
@pytest.mark.parametrize("n_layers", [1, 3, 5])
def test_emission_at_layer_boundaries(dh, n_layers):
    pytest.importorskip("torch")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2405_04229_gb300 import binding as B
    from paper_2405_04229_gb300 import synth
    us = synth.US_STANDARD
    lay = dict(us, **{k: us[k][:n_layers] for k in ("layer_h", "a", "b", "c")})
    lay["h_top"] = us["h_top"] if n_layers == 5 else 60000.0
    edges = [2000.0] + [h for h in lay["layer_h"] if h > 2000.0]
    heights = np.array([e + d for e in edges for d in (0.6 * dh, 1.5 * dh, 12.0, 300.0)])
    segs = synth.shower_segments(len(heights) * 5, 10.0, 0.0, 1e12, seed=3)
    segs["z0"] = np.tile(heights, 5) + 5.0
    segs["inv_gamma2"][:] = np.float32(1e-9)
    atm = B.Atmosphere(layered=lay, refraction=True, transmission=True)
    det = B.Detector(hist=synth.histogram_400(), tel=synth.grid_telescopes())
    g = B.propagate_host(segs, atm, det, seed=5, bunch=1, records=True, snell_dh=dh,
                         record_capacity=4000 * len(heights))
    o = oracle.propagate(segs, oracle.make_atm(oracle.ATM_LAYERED, layered=lay), hist=synth.histogram_400(),
                         tel=synth.grid_telescopes(), bunch=1, refraction=True, transmission=True, seed=5, snell_dh=dh)
    assert PU.compare(g, o, bunch=1)["matched"] > 500


def test_more_slabs_than_a_float_counts():
    """175 km of height in slabs of 1 cm: 1.7e7 slabs, more than 2^24.  In a
    homogeneous medium no slab bends the path: the same ground points as with
    thick slabs, bit for bit."""
    pytest.importorskip("torch")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2405_04229_gb300 import binding as B
    from paper_2405_04229_gb300 import synth
    segs = synth.shower_segments(2, 10.0, 0.0, 1e12, seed=3)
    segs["z0"][:] = 175_000.0
    segs["length"][:] = 1.0
    segs["inv_gamma2"][:] = np.float32(1e-9)
    atm = B.Atmosphere(kind=B.CS_ATM_HOMOGENEOUS, hom_delta=2.9e-4, refraction=True)
    det = B.Detector(hist=synth.histogram_400())
    assert (175_000.0 - 2000.0) / 0.01 > 2**24
    a, b = (B.propagate_host(segs, atm, det, seed=5, bunch=20, records=True, snell_dh=dh) for dh in (0.01, 1000.0))
    assert a["n_records"] == b["n_records"] > 0
    ra, rb = (np.sort(r["records"], order=["seg", "k", "i"]) for r in (a, b))
    for k in ("x", "y", "status"):
        assert np.array_equal(ra[k], rb[k]), k
