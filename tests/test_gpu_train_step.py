"""The fused training step against FP64: loss and gradients at the batch sizes
where its paths begin and end (one block of 256 rows, the reduction's chunk of
256 slices and one beyond), and beside the unfused path at neighbouring sizes."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


# 256: one block; 512, 4352: a few, an odd number; 32768: 256 slices; 33024: a second, partial chunk;
# 255, 257: the unfused path
@pytest.mark.parametrize("rows", [255, 256, 257, 512, 4352, 32768, 33024])
def test_gradients_match_oracle(rows):
    pytest.importorskip("torch")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2405_04229_gb300 import binding as B
    from tests.test_surrogate import _bf16, _split_flat
    rng = np.random.default_rng(rows)
    flat = rng.normal(0, 0.3, oracle.mlp_n_params()).astype(np.float32)
    x = rng.uniform(-1, 1, (rows, 3)).astype(np.float32)
    t = rng.uniform(-1, 1, (rows, 3)).astype(np.float32)
    loss, grad = B.cs_mlp_loss_grad(B.mlp_flat_to_padded(flat), x, t)
    parts = _split_flat(flat.astype(np.float64))
    for k in (2, 4, 6):   # W2..W4 as the tensor cores see them
        parts[k] = _bf16(parts[k]).astype(np.float64)
    loss_o, grad_o = oracle.mlp_loss_grad(np.concatenate(parts), x.astype(np.float64), t.astype(np.float64))
    # BF16 hi + lo operands carry 16 bits, tanh an absolute 2e-7: a relative 2^-14 of each tensor's norm
    assert abs(loss - loss_o) <= 1e-4 * loss_o
    for a, b in zip(_split_flat(B.mlp_padded_to_flat(grad).astype(np.float64)), _split_flat(grad_o)):
        assert np.linalg.norm(a - b) <= 1e-4 * np.linalg.norm(b)
