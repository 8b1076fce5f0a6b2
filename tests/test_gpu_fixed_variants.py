"""The fixed-configuration instances of fluorescence and of the camera optics
against the general ones (which the same call with records runs): whole
numbers equal, time sums to the order of their atomic additions."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

OPT = dict(mirror_d=7.0, focal_f=8.0, camera_r=0.5, point_zenith=0.35, point_azimuth=0.5, cam_n=9)


@pytest.mark.parametrize("spherical", [False, True])
@pytest.mark.parametrize("emission,optics", [(None, OPT), ("half", None), ("half", OPT)])
def test_equal_to_the_general_instance(spherical, emission, optics):
    pytest.importorskip("torch")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2405_04229_gb300 import binding as B
    from paper_2405_04229_gb300 import synth
    segs = synth.shower_segments(3001, 40.0 if spherical else 20.0, 0.0, 1e13, seed=7)
    atm = B.Atmosphere(layered=synth.US_STANDARD, refraction=True, transmission=True, spherical=spherical)
    det = B.Detector(hist=synth.histogram_400(), tel=synth.grid_telescopes(), spherical=spherical, optics=optics)
    kw = dict(fluorescence=dict(synth.FLUORESCENCE, half=True)) if emission else {}
    a, b = (B.propagate_host(segs, atm, det, seed=9, bunch=2, records=rec, **kw) for rec in (False, True))
    assert a["counters"][0] > 0
    if not emission:   # (7,000 photons over the half sphere need not meet a sphere)
        assert a["counters"][B.CS_CNT_TEL] > 0
    for k in ("hist", "tel_counts", "counters") + (("camera",) if optics else ()):
        assert np.array_equal(a[k], b[k]), k
    np.testing.assert_allclose(a["tel_time"], b["tel_time"], rtol=1e-12)
