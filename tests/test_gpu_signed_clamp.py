"""Signed-values rows whose extremes are symmetric: the largest value's code is one above Q_max at some level and is clamped; one element or many
of that value, in calls of many rows and of few."""
import pytest
import torch

from oracle import tsq_ref as R
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


def symmetric_rows(dtype, hidden):
    """A row for every 16-bit value v from 2^-7 to 6: a share of +v that differs from row to row and -v for the rest, then the same number of
    rows of normal values clipped at +v and -v (saturated activations)."""
    first, last = (torch.tensor(t).to(dtype).view(torch.int16).item() for t in (2.0 ** -7, 6.0))
    v = torch.arange(first, last, dtype=torch.int16).view(dtype)[:, None]
    row, col = torch.arange(len(v))[:, None], torch.arange(hidden)[None, :]
    two = torch.where((col * 37 + row) % 11 <= row % 11, v, -v)
    normal = torch.randn((len(v), hidden), generator=torch.Generator().manual_seed(1)) * 2.0 * v.float()
    return torch.cat([two, torch.minimum(torch.maximum(normal, -v.float()), v.float()).to(dtype)]).contiguous()


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16])
@pytest.mark.parametrize("bits", [[4, 8], [2, 4, 8], [2, 3, 4, 8], [3, 6]])
@pytest.mark.parametrize("delta", [0.0, 0.2, 0.35, 0.5])
def test_many_elements_at_the_largest_value(dtype, bits, delta):
    # the largest value's code at the top level may be clamped while a lower level rounds it down: a difference of 1 for each of its elements
    x = symmetric_rows(dtype, 264)
    full_parity(x, 6.0, bits, delta, check_cross=False, variant=1)
    for start in range(0, x.shape[0], x.shape[0] // 5):        # calls of few rows take the other kernel
        full_parity(x[start:start + 8].contiguous(), 6.0, bits, delta, check_cross=False, variant=1)


@pytest.mark.gpu
def test_width_of_a_saturated_row():
    v = torch.full((9, 4096), -0.011474609375, dtype=torch.bfloat16)
    v[:, :1000] = 0.011474609375
    for bits in ([4, 8], [2, 4, 8], [2, 3, 4, 8]):
        blob, _ = full_parity(v, 6.0, bits, 0.2, check_cross=False, variant=1)
        assert set(R.sections(blob)["bits"].tolist()) == {8}
