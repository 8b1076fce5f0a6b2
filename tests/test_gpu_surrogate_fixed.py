"""The surrogate's instances without records (single activations: the fixed
configuration's; split ones: their own) against the ones with records, over
block tiles of every filling: whole numbers equal, time sums to the order of
their additions."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("split", [0, 1])
@pytest.mark.parametrize("spherical", [False, True])
def test_equal_to_the_instance_with_records(spherical, split):
    pytest.importorskip("torch")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2405_04229_gb300 import binding as B
    from paper_2405_04229_gb300 import synth
    atm = B.Atmosphere(layered=synth.US_STANDARD, refraction=True, transmission=True, spherical=spherical)
    det = B.Detector(hist=synth.histogram_400(), tel=synth.grid_telescopes(), spherical=spherical)
    sur = B.Surrogate(atm, epochs=2, n_train=1 << 16, n_heldout=1 << 12, split_activations=split)
    for n in (1, 127, 128, 129, 2003):
        segs = synth.shower_segments(n, 20.0, 0.0, 1e12, seed=n)
        a, b = (B.propagate_host(segs, atm, det, seed=4, bunch=2, records=rec, surrogate=sur) for rec in (False, True))
        assert a["counters"][0] > 0
        for k in ("hist", "tel_counts", "counters"):
            assert np.array_equal(a[k], b[k]), (n, k)
        np.testing.assert_allclose(a["tel_time"], b["tel_time"], rtol=1e-12)
    sur.close()
