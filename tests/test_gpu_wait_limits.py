"""Calls with direct offsets whose waits may run out at any moment: wait limits of a few polls, so that some rows give up while the
rows they wait for are about to publish their sizes.  Either the call says TSQ_ERR_TIMEOUT or its blob is whole, and a workspace
whose call said TSQ_OK is fit for the next call of either kernel."""
import numpy as np
import pytest
import torch

from oracle import tsq_ref as R
from paper_2511_04002_b200 import binding as B
from paper_2511_04002_b200 import synth
from tests._parity import assert_blobs_equal
from tests.test_gpu_parity import rand16

pytestmark = pytest.mark.gpu
OK, TIMEOUT = 0, 7


def whole(plan, x, ws):
    """The call's blob over a known fill (0xA5 where a call writes nothing), compared with the oracle's once."""
    blob = torch.full((plan.sizes(x.shape[0])[0],), 0xA5, dtype=torch.uint8, device="cuda")
    plan.encode(x, blob, ws)
    assert_blobs_equal(blob.cpu().numpy(), R.encode(synth.raw_u16(x.cpu()), R.F16, 6.0, [2, 4, 8], 0.2))
    return blob


@pytest.mark.parametrize("rows_per_sm,hidden", [(1, 4096),     # row = CTA index
                                                (6, 1024),     # rows by ticket, sizes read in batches
                                                (6, 4096), (8, 2048),
                                                (2, 8200)])    # CTAs of more than 256 threads
def test_status_ok_means_a_whole_blob(rows_per_sm, hidden):
    T = rows_per_sm * torch.cuda.get_device_properties(0).multi_processor_count
    plan = B.Plan(torch.float16, hidden, 3000, 6.0, [2, 4, 8], 0.2)
    ws = plan.alloc(1)[1]
    x = rand16((T, hidden), torch.float16, seed=hidden, scale=2.0, outlier_rate=0.01)
    x[1::5] = (x[1::5].float().abs() ** 3 * 0.05).to(torch.float16)  # rows that descend: their sizes come late
    x = x.cuda()
    # a longer call: two kernels
    more = rand16((3000, hidden), torch.float16, seed=3, scale=2.0, outlier_rate=0.01).cuda()
    good, good_more = whole(plan, x, ws), whole(plan, more, ws)
    blob, blob_more = torch.empty_like(good), torch.empty_like(good_more)
    seen = set()
    for k in range(96):
        plan.workspace_set_wait_limit(ws, 1 + k % 32)
        blob.fill_(0xA5)
        plan.encode(x, blob, ws)
        status = plan.blob_info(blob).status
        seen.add(status)
        assert status in (OK, TIMEOUT)
        if status == TIMEOUT:
            assert plan.workspace_status(ws)[0] == TIMEOUT
            plan.workspace_init(ws)
            continue
        assert torch.equal(blob, good), "status 0 with a wait limit of %d, and the blob is not whole" % (1 + k % 32)
        assert plan.workspace_status(ws)[0] == OK
        plan.workspace_set_wait_limit(ws, 0)
        blob.fill_(0xA5)
        blob_more.fill_(0xA5)
        if k % 2:                                              # the next call: the same kernel, then perhaps the other one
            plan.encode(x, blob, ws)
        plan.encode(more, blob_more, ws)
        assert plan.workspace_status(ws)[0] == OK
        assert torch.equal(blob_more, good_more) and (k % 2 == 0 or torch.equal(blob, good))
    print("statuses seen", seen)


def test_a_part_that_gives_up_shows_in_the_host_blob():
    T, H = 2100, 4096                                          # three parts
    plan = B.Plan(torch.float16, H, T, 6.0, [2, 4, 8], 0.2)
    x = rand16((T, H), torch.float16, seed=11, scale=2.0, outlier_rate=0.01)
    x[1::5] = (x[1::5].float().abs() ** 3 * 0.05).to(torch.float16)
    ref = R.encode(synth.raw_u16(x), R.F16, 6.0, [2, 4, 8], 0.2)
    blob, ws = plan.alloc(T)
    x_host, x_dev = x.pin_memory(), torch.empty_like(x, device="cuda")
    blob_host = torch.empty(blob.numel(), dtype=torch.uint8).pin_memory()
    plan.encode_host(x_host, blob_host, x_dev, blob, ws)       # the buffers hold a good blob before every call
    assert_blobs_equal(blob_host.numpy(), ref)
    for k in range(48):
        plan.workspace_set_wait_limit(ws, 1 + k % 32)
        status = OK
        try:
            plan.encode_host(x_host, blob_host, x_dev, blob, ws)
        except B.TsqError as e:
            status = e.status
        assert status in (OK, TIMEOUT)
        assert R.header(blob_host.numpy())["status"] == status and plan.blob_info(blob).status == status
        if status == OK:
            assert_blobs_equal(blob_host.numpy(), ref)
        else:
            plan.workspace_init(ws)
    plan.encode_host(x_host, blob_host, x_dev, blob, ws)
    assert_blobs_equal(blob_host.numpy(), ref)


def test_a_timed_out_part_among_good_ones():
    """Only the first part's wait runs out (row 0 is never handed out); the later parts find their rows and end well."""
    T, H = 2100, 4096
    plan = B.Plan(torch.float16, H, T, 6.0, [2, 4, 8], 0.2)
    x = rand16((T, H), torch.float16, seed=12, scale=2.0, outlier_rate=0.01)
    blob, ws = plan.alloc(T)
    x_host, x_dev = x.pin_memory(), torch.empty_like(x, device="cuda")
    blob_host = torch.zeros(blob.numel(), dtype=torch.uint8).pin_memory()
    plan.workspace_set_wait_limit(ws, 3000)
    torch.cuda.synchronize()
    ws.view(torch.int32)[1] = 1                                # the ticket counter
    torch.cuda.synchronize()
    with pytest.raises(B.TsqError) as e:
        plan.encode_host(x_host, blob_host, x_dev, blob, ws)
    assert e.value.status == TIMEOUT
    assert R.header(blob_host.numpy())["status"] == TIMEOUT and plan.blob_info(blob).status == TIMEOUT
    plan.workspace_init(ws)
    plan.encode_host(x_host, blob_host, x_dev, blob, ws)
    assert_blobs_equal(blob_host.numpy(), R.encode(synth.raw_u16(x), R.F16, 6.0, [2, 4, 8], 0.2))
    assert np.array_equal(blob.cpu().numpy()[:64], blob_host.numpy()[:64])


LAST_GENERATION = (1 << 30) - 2                                # the call that runs as it wipes the descriptors and starts over


@pytest.mark.parametrize("rows_per_sm,hidden", [(1, 1032), (6, 1024), (20, 1024), (1, 8200), (70, 8200)])
def test_generations_start_over(rows_per_sm, hidden):
    # one kernel, rows by index and by ticket, CTAs of up to 256 threads and of more; two kernels, likewise
    T = rows_per_sm * torch.cuda.get_device_properties(0).multi_processor_count
    plan = B.Plan(torch.float16, hidden, T, 6.0, [2, 4, 8], 0.2)
    ws = plan.alloc(1)[1]
    g = torch.Generator(device="cuda").manual_seed(hidden)
    x = (torch.randn((T, hidden), generator=g, device="cuda") * 2.0).to(torch.float16)
    good = whole(plan, x, ws) if rows_per_sm < 70 else torch.full((plan.sizes(T)[0],), 0xA5, dtype=torch.uint8, device="cuda")
    if rows_per_sm == 70:
        plan.encode(x, good, ws)
    torch.cuda.synchronize()
    ws.view(torch.int32)[0] = LAST_GENERATION - 3
    blob = torch.empty_like(good)
    for _ in range(5):                                         # two before it, the call itself, two after
        blob.fill_(0xA5)
        plan.encode(x, blob, ws)
        assert torch.equal(blob, good)
    assert plan.workspace_status(ws) == (OK, OK) and int(ws.view(torch.int32)[0]) == 2


def test_a_wait_that_runs_out_in_the_last_generation():
    T, H = 6 * torch.cuda.get_device_properties(0).multi_processor_count, 1024
    plan = B.Plan(torch.float16, H, T, 6.0, [2, 4, 8], 0.2)
    blob, ws = plan.alloc(T)
    x = torch.randn((T, H), device="cuda").to(torch.float16)
    plan.workspace_set_wait_limit(ws, 3000)
    torch.cuda.synchronize()
    ws.view(torch.int32)[0] = LAST_GENERATION - 1
    ws.view(torch.int32)[1] = 1                                # the ticket counter: row 0 is never handed out
    torch.cuda.synchronize()
    plan.encode(x, blob, ws)
    assert plan.blob_info(blob).status == TIMEOUT and plan.workspace_status(ws)[0] == TIMEOUT
    plan.workspace_init(ws)
    whole(plan, x, ws)
