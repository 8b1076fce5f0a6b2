"""The batch sizes on both sides of the fused training step's upper bound."""
import pytest

from tests.test_gpu_train_step import test_gradients_match_oracle as gradients_match_oracle

pytestmark = pytest.mark.gpu


# 131072 rows: the largest batch of the fused step (1,024 slices); 131328: through global memory
@pytest.mark.parametrize("rows", [131072, 131328])
def test_gradients_match_oracle_at_the_bound(rows):
    gradients_match_oracle(rows)
