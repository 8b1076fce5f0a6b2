"""The planar stepper's pairs of slabs at odd and even numbers of slabs, from
one slab up, with layers left inside a pair and between pairs, against the
FP64 oracle over the same slabs."""
import numpy as np
import pytest

import oracle
from tests import parity_util as PU

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("transmission", [True, False])
@pytest.mark.parametrize("n_slabs", [1, 2, 3, 4, 7])
def test_few_slabs(n_slabs, transmission):
    pytest.importorskip("torch")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2405_04229_gb300 import binding as B
    from paper_2405_04229_gb300 import synth
    segs = synth.shower_segments(400, 20.0, 0.0, 1e12, seed=n_slabs)
    dh = 12000.0 / n_slabs          # emission at 8 to 14 km above the level: n_slabs and its neighbours
    segs["z0"][:] = np.linspace(10000.0, 16000.0, 400)
    segs["inv_gamma2"][:] = np.float32(1e-9)
    atm = B.Atmosphere(layered=synth.US_STANDARD, refraction=True, transmission=transmission)
    det = B.Detector(hist=synth.histogram_400(), tel=synth.grid_telescopes())
    g = B.propagate_host(segs, atm, det, seed=2, bunch=2, records=True, snell_dh=dh)
    o = oracle.propagate(segs, oracle.make_atm(oracle.ATM_LAYERED, layered=synth.US_STANDARD), hist=synth.histogram_400(),
                         tel=synth.grid_telescopes(), bunch=2, refraction=True, transmission=transmission, seed=2, snell_dh=dh)
    assert PU.compare(g, o, bunch=2)["matched"] > 2000
