"""Launches of one round (a tile per resident warp, which starts before the
outputs are zeroed) at the edges of their range: twice in a row the same
outputs, and those of the general instance, which the same call with records
runs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# 152 SMs x 32 warps of tiles of 16 segments at bunch 5: 77,824 segments are the last to fit one round
@pytest.mark.parametrize("n", [1, 31, 4097, 77824, 77825])
@pytest.mark.parametrize("fixed,spherical", [(True, False), (True, True), (False, False)])
def test_equal_to_the_general_instance(n, fixed, spherical):
    pytest.importorskip("torch")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2405_04229_gb300 import binding as B
    from paper_2405_04229_gb300 import synth
    segs = synth.shower_segments(n, 20.0, 0.0, 1e12, seed=n)
    atm = B.Atmosphere(layered=synth.US_STANDARD, refraction=fixed, transmission=fixed, spherical=spherical)
    det = B.Detector(hist=synth.histogram_400(), tel=synth.grid_telescopes() if fixed else None, spherical=spherical)
    kw = dict(seed=6, bunch=5)
    a, b = B.propagate_host(segs, atm, det, **kw), B.propagate_host(segs, atm, det, **kw)
    r = B.propagate_host(segs, atm, det, records=True, record_capacity=1024 + 30 * n, **kw)
    assert a["counters"][B.CS_CNT_EMITTED] > 0
    for k in ("hist", "tel_counts", "counters"):
        assert np.array_equal(a[k], b[k]) and np.array_equal(a[k], r[k]), k
    for o in (b, r):
        np.testing.assert_allclose(a["tel_time"], o["tel_time"], rtol=1e-12)
