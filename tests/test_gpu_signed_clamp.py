"""Signed-values rows whose extremes both touch the threshold: the largest value's code is one above Q_max and is clamped."""
import pytest
import torch

from tests._parity import full_parity
from tests.test_gpu_parity import rand16


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16])
@pytest.mark.parametrize("shape", [(1000, 4096), (1100, 1032), (960, 8184)])
@pytest.mark.parametrize("delta", [0.2, 0.45, 1e9])
def test_rows_with_symmetric_extremes(dtype, shape, delta):
    x = rand16(shape, dtype, seed=shape[1], scale=1.5, outlier_rate=0.01)
    top = torch.tensor(6.0).to(dtype)
    below = (top.view(torch.int16) - 1).view(dtype)                  # the largest value below the threshold
    x[:, 3], x[:, 5] = below, -below
    x[::3] = x[::3].abs()
    x[1::6, 1::2] *= 0.01
    full_parity(x, 6.0, [2, 3, 4, 8], delta, check_cross=False, variant=1)
