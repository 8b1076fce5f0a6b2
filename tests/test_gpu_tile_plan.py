"""The launch plan's tile sizes and parts do not change a result: one call over
n segments (tiles of 1 to 32 segments, the stepper's rounds dealt out in parts)
gives the counts of the same segments handed over in small pieces."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    pytest.importorskip("torch")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2405_04229_gb300 import binding as B
    from paper_2405_04229_gb300 import synth
    return B, synth


# tile sizes of the plan: 1 (n = 1, 33, 257), 1 and 2 (1001), 2 and 4 (5003), 4 and 8 (20011)
@pytest.mark.parametrize("n", [1, 33, 257, 1001, 5003, 20011])
@pytest.mark.parametrize("bunch", [1, 5])
@pytest.mark.parametrize("snell_dh,spherical", [(None, False), (None, True), (200.0, False)])
def test_one_call_equals_pieces(lib, n, bunch, snell_dh, spherical):
    B, synth = lib
    segs = B.pack_segments(synth.shower_segments(n, 20.0, 0.0, 1e12, seed=11))
    segs["length"][: max(1, n // 50)] = 90.0   # more sub-steps and bunches than one round and one window hold
    atm = B.Atmosphere(layered=synth.US_STANDARD, refraction=True, transmission=True, spherical=spherical)
    det = B.Detector(hist=synth.histogram_400(), tel=synth.grid_telescopes(), spherical=spherical)
    kw = dict(seed=4, bunch=bunch, snell_dh=snell_dh)
    one = B.propagate_host(segs, atm, det, **kw)
    piece = max(n // 7, 1)
    parts = [B.propagate_host(segs[a:a + piece], atm, det, seg_base=a, **kw) for a in range(0, n, piece)]
    for k in ("hist", "tel_counts", "counters"):
        assert np.array_equal(one[k], sum(p[k] for p in parts)), k
    assert one["counters"][B.CS_CNT_EMITTED] > 0
    np.testing.assert_allclose(one["tel_time"], sum(p["tel_time"] for p in parts), rtol=1e-12)
