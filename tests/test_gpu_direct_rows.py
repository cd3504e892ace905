"""Calls of a few rows per SM (one kernel, offsets read directly, last row's CTA ends the call) at the edges of their range, several on one
workspace, mixed with calls of two kernels."""
import numpy as np
import pytest
import torch

from oracle import tsq_ref as R
from paper_2511_04002_b200 import binding as B
from paper_2511_04002_b200 import synth
from tests._parity import assert_blobs_equal, gpu_decode, gpu_encode
from tests.test_gpu_parity import rand16

pytestmark = pytest.mark.gpu


def longest_call_of_one_kernel(plan, x, blob, ws):
    """Rows of the longest call that takes one launch: asked of the library, which knows its kernels' occupancy."""
    def launches(T):
        before = B.kernel_launch_count()
        plan.encode(x[:T], blob, ws)
        return B.kernel_launch_count() - before

    one, two = 1, x.shape[0]
    assert launches(one) == 1 and launches(two) == 2
    while two - one > 1:
        T = (one + two) // 2
        one, two = (T, two) if launches(T) == 1 else (one, T)
    return one


@pytest.mark.parametrize("hidden", [8, 1032, 4096, 16384])
def test_edges_of_the_range_on_one_workspace(hidden):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    sizes = [1, 2, sms - 1, sms, sms + 1, 2 * sms + 1, 6 * sms, 6 * sms + 1, 8 * sms, 8 * sms + 1, 3]
    plan = B.Plan(torch.float16, hidden, max(sizes), 6.0, [2, 4, 8], 0.2)
    ws = plan.alloc(1)[1]
    for k, T in enumerate(sizes):
        x = rand16((T, hidden), torch.float16, seed=hidden + k, scale=2.0, outlier_rate=0.01)
        x[::3] = (x[::3].float().abs() * 0.2).to(torch.float16)          # rows without outliers
        x[1::5] = (x[1::5].float().abs() ** 3 * 0.05).to(torch.float16)  # rows that descend
        blob = torch.zeros(plan.sizes(T)[0], dtype=torch.uint8, device="cuda")
        _, got, _ = gpu_encode(plan, x, ws=ws, blob=blob)
        ref = R.encode(synth.raw_u16(x), R.F16, 6.0, [2, 4, 8], 0.2)
        assert_blobs_equal(got, ref)
        assert np.array_equal(gpu_decode(plan, blob, T, ws), R.decode(ref))
    assert plan.workspace_status(ws) == (0, 0)


def test_many_calls_back_to_back_on_one_stream():
    # launches overlap their predecessors: every call reads what the one before it wrote
    T, H = 64, 4096
    plan = B.Plan(torch.bfloat16, H, T, 6.0, [2, 4, 8], 0.2)
    blob, ws = plan.alloc(T)
    x = rand16((T, H), torch.bfloat16, seed=1, scale=2.0, outlier_rate=0.01).cuda()
    y = torch.empty_like(x)
    want = None
    for i in range(300):
        plan.encode(x if i == 0 else y, blob, ws)        # encodes what the last call decoded
        plan.decode(blob, T, y, ws)
        if i == 0:
            want = y.clone()
    torch.cuda.synchronize()
    assert plan.workspace_status(ws) == (0, 0)
    cpu = want.cpu()
    for _ in range(299):
        nxt = synth.from_raw_u16(R.decode(R.encode(synth.raw_u16(cpu), R.BF16, 6.0, [2, 4, 8], 0.2)), "bf16")
        if torch.equal(nxt.view(torch.int16), cpu.view(torch.int16)):
            break
        cpu = nxt
    assert torch.equal(y.cpu().view(torch.int16), cpu.view(torch.int16))


@pytest.mark.parametrize("bits", [[2, 4, 8], [2, 3, 6]])
@pytest.mark.parametrize("dtype,hidden", [(torch.float16, 1032), (torch.bfloat16, 5120)])
def test_every_instance_and_the_line_to_the_two_kernels(dtype, hidden, bits):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    plan = B.Plan(dtype, hidden, 14 * sms + 1, 6.0, bits, 0.2)
    blob, ws = plan.alloc(14 * sms + 1)
    x = rand16((14 * sms + 1, hidden), dtype, seed=hidden, scale=2.0, outlier_rate=0.01)
    x[::3] = (x[::3].float().abs() * 0.2).to(dtype)              # rows without outliers
    x[1::5] = (x[1::5].float().abs() ** 3 * 0.05).to(dtype)      # rows that descend
    x[7::29] = (x[7::29].float().abs() * 0.1 + 3.0).to(dtype)    # rows that need the division instruction
    line = longest_call_of_one_kernel(plan, x.cuda(), blob, ws)
    # with rows of 5120 elements an SM holds 3, 4 and 6 CTAs of the three instances
    for T in (3 * sms + 5, 4 * sms + 9, 5 * sms, line, line + 1, 9 * sms, 14 * sms + 1):
        blob = torch.zeros(plan.sizes(T)[0], dtype=torch.uint8, device="cuda")
        _, got, _ = gpu_encode(plan, x[:T], ws=ws, blob=blob)
        assert_blobs_equal(got, R.encode(synth.raw_u16(x[:T]), R.F16 if dtype == torch.float16 else R.BF16, 6.0, bits, 0.2))
    assert plan.workspace_status(ws) == (0, 0)


@pytest.mark.parametrize("hidden,signed", [(8200, False), (8200, True)])
def test_long_rows_and_the_line_to_the_two_kernels(hidden, signed):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    variant = B.VARIANT_SIGNED_VALUES if signed else B.VARIANT_MAGNITUDES
    plan = B.Plan(torch.bfloat16, hidden, 64 * sms + 1, 6.0, [2, 4, 8], 0.2, variant=variant)
    blob, ws = plan.alloc(64 * sms + 1)
    x = rand16((64 * sms + 1, hidden), torch.bfloat16, seed=7, scale=2.0, outlier_rate=0.01)
    x[::3] = (x[::3].float().abs() * 0.2).to(torch.bfloat16)
    x = x.cuda()
    line = longest_call_of_one_kernel(plan, x, blob, ws)
    for T in (line, line + 1, 7 * sms + 1):
        _, got, _ = gpu_encode(plan, x[:T].cpu(), ws=ws)
        if T <= line + 1 or not signed:
            assert_blobs_equal(got, R.encode(synth.raw_u16(x[:T].cpu()), R.BF16, 6.0, [2, 4, 8], 0.2, signed_values=signed))
    # the rows of a call of one kernel decode as in calls of two
    y = [torch.empty_like(x) for _ in range(3)]
    sizes = (line, line + 1, 64 * sms + 1)
    for k, T in enumerate(sizes):
        plan.encode(x[:T], blob, ws)
        plan.decode(blob, T, y[k][:T], ws)
    assert plan.workspace_status(ws) == (0, 0)
    for k in (0, 1):
        assert torch.equal(y[k][:sizes[k]].view(torch.int16), y[k + 1][:sizes[k]].view(torch.int16))


def test_a_wait_that_runs_out_ends_a_call_of_many_turns():
    # row 0 is never produced.  Two kernels, which wait for nothing: the call ends at once.  Parts of a host-buffer call, one kernel each and the
    # longest calls of it, in several turns of CTAs: one limit's worth of waiting for the part, not one for each turn
    T, H = 30 * torch.cuda.get_device_properties(0).multi_processor_count, 8200
    plan = B.Plan(torch.bfloat16, H, T, 6.0, [2, 4, 8], 0.2)
    blob, ws = plan.alloc(T)
    x = torch.randn((T, H), device="cuda").to(torch.bfloat16)
    plan.workspace_set_wait_limit(ws, 3000)
    ws.view(torch.int32)[1] = 1  # the ticket counter
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    plan.encode(x, blob, ws)
    e1.record()
    torch.cuda.synchronize()
    assert plan.workspace_status(ws)[0] == 7 and plan.blob_info(blob).status == 7
    assert e0.elapsed_time(e1) < 40.0
    plan.workspace_init(ws)
    plan.workspace_set_wait_limit(ws, 3000)
    ws.view(torch.int32)[1] = 1
    x_host = x.cpu().pin_memory()
    blob_host = torch.empty(blob.numel(), dtype=torch.uint8).pin_memory()
    e0.record()
    with pytest.raises(B.TsqError) as e:
        plan.encode_host(x_host, blob_host, x, blob, ws)
    e1.record()
    torch.cuda.synchronize()
    assert e.value.status == 7 and plan.workspace_status(ws)[0] == 7 and e0.elapsed_time(e1) < 40.0
    plan.workspace_init(ws)
    _, got, _ = gpu_encode(plan, x[:5].cpu(), ws=ws)
    assert_blobs_equal(got, R.encode(synth.raw_u16(x[:5].cpu()), R.BF16, 6.0, [2, 4, 8], 0.2))
