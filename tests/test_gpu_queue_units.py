"""The exact pass's queue beyond one unit of 256 entries a block: the block
orders each unit by height in shared memory that the unit before has used.
More entries than the grid's blocks take in one turn, on the plane and the
sphere, against the tile map, which has no queue."""
import numpy as np
import pytest

from paper_2405_04229_gb300 import binding as B
from paper_2405_04229_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("spherical", [False, True])
def test_second_turn_of_the_queue(spherical):
    import __graft_entry__
    __graft_entry__.build()
    segs = synth.shower_segments(400_000, 30.0, 30.0, 1e13, seed=32)
    fl = dict(synth.FLUORESCENCE, half=True)
    atm = B.Atmosphere(layered=synth.US_STANDARD, refraction=True, transmission=True, spherical=spherical)
    det = B.Detector(hist=synth.histogram_400(), tel=synth.grid_telescopes(), spherical=spherical)
    queue, tiles = (B.propagate_host(segs, atm, det, seed=4, bunch=1, fluorescence=fl, exact_queue=q) for q in (0, -1))
    # of light emitted evenly into the lower half sphere cos 75 deg lies beyond the tables: more than a
    # turn of 4 blocks an SM, and less than the default queue's 32 entries a tile (one a segment)
    beyond = 0.2588 * int(queue["counters"][B.CS_CNT_EMITTED])
    assert 1.1 * 4 * 256 * B.cs_device_sm_count() < beyond < 0.9 * len(segs["z0"])
    for k in ("hist", "tel_counts", "counters"):
        assert np.array_equal(queue[k], tiles[k]), k
    np.testing.assert_allclose(queue["tel_time"], tiles["tel_time"], rtol=1e-12)
    assert int(queue["counters"][B.CS_CNT_TEL]) > 0
