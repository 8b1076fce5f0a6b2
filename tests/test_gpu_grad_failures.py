"""cs_mlp_loss_grad reports a tensor-core wait that gave up and a copy that
failed; it does not return gradients with CS_OK.  Both batch forms: 256 rows
through the fused step, 255 through global memory."""
import numpy as np
import pytest

from paper_2405_04229_gb300 import binding as B
from tests import fake_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    with fake_cuda.loaded(fake_cuda.link(str(tmp_path_factory.mktemp("fake")))) as f:
        yield f


def _call(rows):
    rng = np.random.default_rng(rows)
    params = rng.normal(0, 0.3, B.N_MLP_PARAMS).astype(np.float32)
    x, t = (rng.uniform(-1, 1, (rows, 3)).astype(np.float32) for _ in range(2))
    grad, loss = np.zeros_like(params), np.zeros(1, np.float32)
    st = B.lib().cs_mlp_loss_grad(B._dptr(params), B._dptr(x), B._dptr(t), rows, B._dptr(grad), B._dptr(loss))
    return st, grad


@pytest.mark.parametrize("rows", [255, 256])
def test_give_up_is_reported(fake, rows):
    fake.reset(timed_out=1)
    assert _call(rows)[0] == B.CS_ERR_TIMEOUT
    fake.reset()
    st, grad = _call(rows)   # the flag was taken: the next call succeeds
    assert st == B.CS_OK and np.any(grad != 0.0)


@pytest.mark.parametrize("rows", [255, 256])
def test_failed_copy_is_reported(fake, rows):
    fake.reset()
    assert _call(rows)[0] == B.CS_OK
    n = fake.copies
    assert n >= 5   # samples, targets, parameters; gradients, loss
    for k in range(n):
        fake.reset(fail_copy=k)
        assert _call(rows)[0] == B.CS_ERR_CUDA, k
