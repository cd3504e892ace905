"""The two-kernel encoder in calls of many rows: both sides of the line where pack_kernel's threads take 64 elements instead of 32 (80
segments of 1024 elements per SM; rows of one segment always 32, rows of more than five always 64), each way of deciding the first lower
candidate, whole and ragged groups."""
import numpy as np
import pytest
import torch

from oracle import tsq_ref as R
from paper_2511_04002_b200 import binding as B
from paper_2511_04002_b200 import synth
from tests._parity import assert_blobs_equal, full_parity, gpu_decode, gpu_encode
from tests.test_gpu_parity import rand16

pytestmark = pytest.mark.gpu


def rows_at_the_line(hidden):
    return 80 * torch.cuda.get_device_properties(0).multi_processor_count // max(2, (hidden + 1023) // 1024)


@pytest.mark.parametrize("bits", [[2, 4, 8], [2, 3, 6]])
@pytest.mark.parametrize("dtype,hidden", [(torch.float16, 8), (torch.bfloat16, 1032), (torch.float16, 2048), (torch.bfloat16, 5120)])
def test_both_sides_of_the_line(dtype, hidden, bits):
    line = rows_at_the_line(hidden)
    plan = B.Plan(dtype, hidden, line + 3, 6.0, bits, 0.2)
    ws = plan.alloc(1)[1]
    x = rand16((line + 3, hidden), dtype, seed=hidden, scale=2.0, outlier_rate=0.002)
    x[::3] = (x[::3].float().abs() * 0.2).to(dtype)           # rows without outliers
    x[1::17] = (x[1::17].float().abs() ** 3 * 0.05).to(dtype)  # rows that descend
    x[5::301] = (x[5::301].float() * 4.0).to(dtype)            # rows that are mostly outliers
    x[7::299] = (x[7::299].float().abs() * 0.1 + 3.0).to(dtype)  # rows that need the division instruction
    for T in (line, line + 1, line + 3):
        blob = torch.zeros(plan.sizes(T)[0], dtype=torch.uint8, device="cuda")
        _, got, _ = gpu_encode(plan, x[:T], ws=ws, blob=blob)
        ref = R.encode(synth.raw_u16(x[:T]), R.F16 if dtype == torch.float16 else R.BF16, 6.0, bits, 0.2)
        assert_blobs_equal(got, ref)
        if T == line:
            assert np.array_equal(gpu_decode(plan, blob, T, ws), R.decode(ref))
    assert plan.workspace_status(ws) == (0, 0)


@pytest.mark.parametrize("dtype,hidden", [(torch.float16, 2048), (torch.bfloat16, 1032)])
def test_signed_values(dtype, hidden):
    line = rows_at_the_line(hidden)
    x = rand16((line + 1, hidden), dtype, seed=hidden, scale=2.0, outlier_rate=0.002)
    x[::3] = (x[::3].float().abs() * 0.2).to(dtype)
    x[7::299] = (x[7::299].float().abs() * 0.1 + 3.0).to(dtype)
    full_parity(x, 6.0, [2, 4, 8], 0.2, check_cross=False, variant=1)


@pytest.mark.parametrize("bits", [[2, 4, 8], [8]])
@pytest.mark.parametrize("dtype,hidden", [(torch.float16, 1032), (torch.bfloat16, 5120)])
def test_signed_values_ragged_fp16_and_whole_bf16_groups(dtype, hidden, bits):
    # with the cases above: signed rows of both types with whole and with short last groups, each over every kind of row
    line = rows_at_the_line(hidden)
    x = rand16((line + 1, hidden), dtype, seed=hidden + 1, scale=2.0, outlier_rate=0.002)
    x[::3] = (x[::3].float().abs() * 0.2).to(dtype)
    x[1::17] = (x[1::17].float().abs() ** 3 * 0.05).to(dtype)
    x[5::301] = (x[5::301].float() * 4.0).to(dtype)
    x[7::299] = (x[7::299].float().abs() * 0.1 + 3.0).to(dtype)
    full_parity(x, 6.0, bits, 0.2, check_cross=False, variant=1)
