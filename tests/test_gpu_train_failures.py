"""cs_surrogate_train reports each copy of its own that fails: no network comes
back whose constants or held-out errors were never copied."""
import ctypes as C

import pytest

from paper_2405_04229_gb300 import binding as B
from paper_2405_04229_gb300 import synth
from tests import fake_cuda

pytestmark = pytest.mark.gpu

# heights, columns, baseline, range, initial parameters, schedule, loss, trained parameters, four arrays
# of held-out labels, evaluation inputs, evaluation outputs
COPIES = 14


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    with fake_cuda.loaded(fake_cuda.link(str(tmp_path_factory.mktemp("fake")))) as f:
        f.atm = B.Atmosphere(layered=synth.US_STANDARD, refraction=True, transmission=True)
        yield f
        f.atm.close()


def _train(fake, **how):
    c = B.cs_surrogate_config()
    B.lib().cs_surrogate_config_default(C.byref(c))
    c.n_train, c.n_heldout, c.batch, c.epochs = 4096, 64, 1024, 1
    h, st = C.c_void_p(), B.cs_surrogate_stats()
    fake.reset(**how)
    status = B.lib().cs_surrogate_train(fake.atm.handle, C.byref(c), C.byref(h), C.byref(st))
    made = bool(h.value)
    if made:
        B.lib().cs_surrogate_destroy(h)
    return status, made


def test_undisturbed_training_makes_these_copies(fake):
    assert _train(fake) == (B.CS_OK, True)
    assert fake.copies == COPIES


@pytest.mark.parametrize("k", range(COPIES))
def test_failed_copy_is_reported(fake, k):
    assert _train(fake, fail_copy=k) == (B.CS_ERR_CUDA, False)


def test_give_up_is_reported(fake):
    assert _train(fake, timed_out=1) == (B.CS_ERR_TIMEOUT, False)
    assert _train(fake) == (B.CS_OK, True)
