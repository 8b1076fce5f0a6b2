"""A call that does not accumulate starts from zero whatever its buffers held,
at odd sizes and at buffers aligned to 8 bytes only, and writes nothing beyond
them; a call that accumulates adds to them."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [0, 1, 700])
@pytest.mark.parametrize("cells,n_tel,cam_n", [((1, 1), 1, 0), ((3, 7), 0, 0), ((41, 37), 3, 5), ((256, 64), 4, 0)])
@pytest.mark.parametrize("offset", [0, 1])
def test_outputs_start_from_zero(n, cells, n_tel, cam_n, offset):
    torch = pytest.importorskip("torch")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2405_04229_gb300 import binding as B
    from paper_2405_04229_gb300 import synth
    segs = B.pack_segments(synth.shower_segments(max(n, 1), 20.0, 0.0, 1e12, seed=2))[:n]
    nx, ny = cells
    hist = dict(nx=nx, ny=ny, x0=-150.0, y0=-150.0, dx=300.0 / nx, dy=300.0 / ny)
    optics = dict(mirror_d=7.0, focal_f=8.0, camera_r=0.5, point_zenith=0.35, point_azimuth=0.0, cam_n=cam_n)
    atm = B.Atmosphere(layered=synth.US_STANDARD, refraction=True, transmission=True)
    det = B.Detector(n_showers=3, hist=hist, tel=synth.grid_telescopes(nx=n_tel, ny=1, pitch=30.0) if n_tel else None,
                     optics=optics if cam_n else None)
    sizes = dict(hist=3 * nx * ny, tel_counts=3 * n_tel, tel_time=3 * n_tel, counters=8, record_count=1,
                 camera=3 * n_tel * cam_n * cam_n)
    d = torch.from_numpy(segs.view(np.uint8).copy()).cuda()

    def call(accumulate, garbage):
        buf = {k: torch.full((v + 4,), garbage, dtype=torch.int64, device="cuda") for k, v in sizes.items()}
        view = {k: buf[k][offset:offset + v] for k, v in sizes.items()}
        out = B.cs_output()
        for k, v in sizes.items():
            if v:
                setattr(out, k, view[k].data_ptr())
        o = B.cs_opts_default()
        o.bunch, o.device_ptrs, o.accumulate = 5, 1, accumulate
        st = B.cs_propagate_ex(C.c_void_p(d.data_ptr()) if n else None, n, atm.handle, det.handle, 1, o, out, B.stream_ptr())
        assert st == B.CS_OK
        torch.cuda.synchronize()
        for k, v in sizes.items():   # the words around each buffer are untouched
            assert bool((buf[k][:offset] == garbage).all()) and bool((buf[k][offset + v:] == garbage).all()), k
        return {k: v.cpu().numpy() for k, v in view.items()}

    fresh, dirty, added = call(0, 0), call(0, 0x7F11223344556677), call(1, 100)
    for k in ("hist", "tel_counts", "counters", "record_count", "camera"):
        assert np.array_equal(fresh[k], dirty[k]), k
        if k != "record_count":
            assert np.array_equal(fresh[k] + 100, added[k]), k
    np.testing.assert_allclose(dirty["tel_time"].view(np.float64), fresh["tel_time"].view(np.float64), rtol=1e-12)
    assert (fresh["counters"][0] > 0) == (n > 0)
