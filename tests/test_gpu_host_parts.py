"""Host-buffer calls large enough to go in parts: the same bytes as the device calls give, at ragged sizes, for parts that
end in the middle of a call's last rows, and with an outlier capacity that runs out in a later part."""
import numpy as np
import pytest
import torch

from oracle import tsq_ref as R
from paper_2511_04002_b200 import binding as B
from paper_2511_04002_b200 import synth
from tests._parity import assert_blobs_equal
from tests.test_gpu_parity import rand16

pytestmark = pytest.mark.gpu


def host_call(plan, x):
    T = x.shape[0]
    blob, ws = plan.alloc(T)
    blob.fill_(0xA5)
    blob_host = torch.full((blob.numel(),), 0x5A, dtype=torch.uint8).pin_memory()
    x_dev = torch.empty_like(x, device="cuda")
    status = 0
    try:
        payload = plan.encode_host(x.pin_memory(), blob_host, x_dev, blob, ws)
        assert payload == plan.blob_info(blob).payload_bytes
    except B.TsqError as e:
        status = e.status
    return blob_host, blob, ws, status


@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16])
@pytest.mark.parametrize("shape", [(2048, 2048), (2053, 2056), (2048, 4096), (1000, 16384), (70, 65536), (7111, 1000)])
def test_parts_give_the_device_calls_bytes(dtype, shape, variant):
    x = rand16(shape, dtype, seed=shape[0] + shape[1], scale=2.0, outlier_rate=0.01)
    x[::7] = (x[::7].float().abs() ** 3 * 0.05).to(dtype)
    plan = B.Plan(dtype, shape[1], shape[0], 6.0, [2, 4, 8], 0.2, variant=variant)
    blob_host, blob, ws, status = host_call(plan, x)
    assert status == 0
    ref = R.encode(synth.raw_u16(x), R.F16 if dtype == torch.float16 else R.BF16, 6.0, [2, 4, 8], 0.2, signed_values=variant == 1)
    assert_blobs_equal(blob_host.numpy(), ref)
    y = torch.full_like(x, 7.0).pin_memory()
    y_dev = torch.empty_like(x, device="cuda")
    plan.decode_host(blob_host, shape[0], y, blob, y_dev, ws)
    assert np.array_equal(synth.raw_u16(y), R.decode(ref))
    assert plan.workspace_status(ws) == (0, 0)


def test_capacity_that_runs_out_and_a_blob_that_lies_about_its_offsets():
    T, H = 1024, 4096                              # two parts of 512 rows
    x = rand16((T, H), torch.float16, seed=5, scale=2.0, outlier_rate=0.01)
    plan = B.Plan(torch.float16, H, T, 6.0, [2, 4, 8], 0.2, max_outliers=20000)
    blob_host, blob, ws, status = host_call(plan, x)
    ref = R.encode(synth.raw_u16(x), R.F16, 6.0, [2, 4, 8], 0.2, 20000)
    assert status == 6 and R.header(ref)["status"] == 6
    assert_blobs_equal(blob_host.numpy(), ref)
    plan = B.Plan(torch.float16, H, T, 6.0, [2, 4, 8], 0.2)
    blob_host, blob, ws, status = host_call(plan, x)
    assert status == 0
    lay = R.layout(H, T, 8, 0)
    at = lay["word_off"] + 4 * 512
    bad = blob_host.clone().pin_memory()
    bad[at:at + 4] = 255
    y, y_dev = torch.zeros_like(x).pin_memory(), torch.empty_like(x, device="cuda")
    with pytest.raises(B.TsqError) as e:
        plan.decode_host(bad, T, y, blob, y_dev, ws)
    assert e.value.status == 5
