"""The evaluation kernel's block sizes (128, 256 and 512 points at the edges of
their ranges): every point's fields as in one call over all of them."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("split", [0, 1])
def test_block_sizes_agree(split):
    torch = pytest.importorskip("torch")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2405_04229_gb300 import binding as B
    from paper_2405_04229_gb300 import synth
    atm = B.Atmosphere(layered=synth.US_STANDARD, refraction=True, transmission=True)
    sur = B.Surrogate(atm, epochs=1, n_train=1 << 15, n_heldout=1 << 12, split_activations=split)
    n = 100_003
    g = torch.Generator().manual_seed(5)
    x = torch.rand(n, 4, generator=g)
    x = (x * torch.tensor([25000.0, 0.45, 1.6e-3, 0.0]) + torch.tensor([100.0, 0.55, 1.7e-3, 0.0])).cuda()
    out = torch.zeros(n, 4, device="cuda")

    def run(m, o):
        st = B.lib().cs_surrogate_eval(sur.handle, C.c_void_p(x.data_ptr()), m, C.c_void_p(o.data_ptr()), B.stream_ptr())
        assert st == B.CS_OK
    run(n, out)
    assert bool(torch.isfinite(out).all()) and float(out.abs().max()) > 0
    for m in (1, 127, 129, 152 * 128, 152 * 128 + 1, 304 * 128, 304 * 128 + 1, 304 * 256, 304 * 256 + 1):
        part = torch.zeros(n, 4, device="cuda")
        run(m, part)
        assert np.array_equal(part[:m].cpu().numpy(), out[:m].cpu().numpy()), m
        assert not bool(part[m:].any()), m
    sur.close()
