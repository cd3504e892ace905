"""The two-kernel encoder where its blocks of rows end, at the edges of its thread shapes, with rows that stop at every candidate, with magnitudes
that lie on a rounding boundary, and on one workspace with calls of other sizes and of the one-kernel encoder."""
import numpy as np
import pytest
import torch

from oracle import tsq_ref as R
from paper_2511_04002_b200 import binding as B
from paper_2511_04002_b200 import synth
from tests._parity import assert_blobs_equal, gpu_decode
from tests.test_gpu_parity import rand16

pytestmark = pytest.mark.gpu


def rows_of_every_kind(tokens, hidden, dtype, seed):
    x = rand16((tokens, hidden), dtype, seed=seed, scale=2.0, outlier_rate=0.004)
    x[::3] = (x[::3].float().abs() * 0.2 + 0.01).to(dtype)          # no outlier, a smallest magnitude above 0
    x[1::7] = (x[1::7].float().abs() ** 3 * 0.05).to(dtype)         # rows that descend
    x[2::31] = (x[2::31].float() * 9.0).to(dtype)                   # mostly outliers: longer than a warp's list
    x[3::37] = (x[3::37].float().abs() * 0.1 + 3.0).to(dtype)       # the division instruction
    g = torch.Generator().manual_seed(seed)
    k = torch.randint(0, 15, (len(x[4::11]), hidden), generator=g).float()
    x[4::11] = (k * 7.0 / 14.0 * 0.75).to(dtype)                    # on the boundaries of the 4-bit level: multiples of hi / 14
    x[5::13] = torch.where(x[5::13].float().abs() < 1.0, 2.0, 4.0).to(dtype)  # half and whole of the largest magnitude
    x[6::41] = 0.0
    return x


def check(plan, x, ws, bits, variant=0, fill=0xA5, delta=0.2):
    T = x.shape[0]
    blob = torch.full((plan.sizes(T)[0],), fill, dtype=torch.uint8, device="cuda")
    plan.encode(x.cuda(), blob, ws)
    ref = R.encode(synth.raw_u16(x), R.F16 if x.dtype == torch.float16 else R.BF16, 6.0, bits, delta, signed_values=variant == 1)
    assert_blobs_equal(blob.cpu().numpy(), ref)
    return blob, ref


@pytest.mark.parametrize("bits", [[2, 4, 8], [2, 3, 4, 8], [3, 4, 8], [4, 8], [2, 3, 6]])
@pytest.mark.parametrize("dtype,hidden", [(torch.float16, 8), (torch.bfloat16, 1000), (torch.float16, 1288), (torch.bfloat16, 4096),
                                          (torch.float16, 5120), (torch.bfloat16, 8200), (torch.float16, 10248)])
def test_every_kind_of_row(dtype, hidden, bits):
    T = 6 * torch.cuda.get_device_properties(0).multi_processor_count + 1
    plan = B.Plan(dtype, hidden, T, 6.0, bits, 0.2)
    ws = plan.alloc(1)[1]
    x = rows_of_every_kind(T, hidden, dtype, hidden)
    blob, ref = check(plan, x, ws, bits)
    if bits == [2, 4, 8]:
        assert np.array_equal(gpu_decode(plan, blob, T, ws), R.decode(ref))
    assert plan.workspace_status(ws) == (0, 0)


@pytest.mark.parametrize("delta", [-1.0, 0.0, 0.05, 1e9])
def test_other_tolerances(delta):
    T, H, bits = 6 * torch.cuda.get_device_properties(0).multi_processor_count + 1, 2048, [2, 3, 4, 8]
    plan = B.Plan(torch.float16, H, T, 6.0, bits, delta)
    check(plan, rows_of_every_kind(T, H, torch.float16, 9), plan.alloc(1)[1], bits, delta=delta)


@pytest.mark.parametrize("hidden,variant", [(16384, 0), (16392, 0), (65536, 0), (16384, 1), (16392, 1)])
def test_long_rows(hidden, variant):
    T = (2 if variant == 0 else 6) * torch.cuda.get_device_properties(0).multi_processor_count + 1
    plan = B.Plan(torch.bfloat16, hidden, T, 6.0, [2, 4, 8], 0.2, variant=variant)
    check(plan, rows_of_every_kind(T, hidden, torch.bfloat16, hidden), plan.alloc(1)[1], [2, 4, 8], variant)


def test_blocks_of_rows_and_calls_of_other_sizes_on_one_workspace():
    # sums of 32, 1024 and 32768 rows: calls that end on, before and after a block, longer and shorter ones in turn, so that every call meets
    # the cells that others have used; between them calls of one kernel, and a plan of fewer tokens on the same workspace
    H, bits = 16, [2, 4, 8]
    big, small = B.Plan(torch.float16, H, 66000, 6.0, bits, 0.2), B.Plan(torch.float16, H, 2050, 6.0, bits, 0.2)
    ws = big.alloc(1)[1]
    x = rows_of_every_kind(66000, H, torch.float16, 3)
    for k, T in enumerate((66000, 1024, 100, 32768, 1023, 65537, 1025, 5, 32767, 2048, 32769, 66000, 65536)):
        check(small if T <= 2050 and k % 2 else big, x[:T], ws, bits, fill=k)
    assert big.workspace_status(ws) == (0, 0)


def test_capacity_that_runs_out():
    T, H = 1500, 1024
    plan = B.Plan(torch.float16, H, T, 6.0, [2, 4, 8], 0.2, max_outliers=3000)
    x = rand16((T, H), torch.float16, seed=2, scale=2.0, outlier_rate=0.01)
    ws = plan.alloc(1)[1]
    blob = torch.full((plan.sizes(T)[0],), 0xA5, dtype=torch.uint8, device="cuda")
    plan.encode(x.cuda(), blob, ws)
    ref = R.encode(synth.raw_u16(x), R.F16, 6.0, [2, 4, 8], 0.2, 3000)
    assert plan.blob_info(blob).status == 6 == R.header(ref)["status"] and plan.workspace_status(ws)[0] == 6
    assert_blobs_equal(blob.cpu().numpy(), ref)


def test_under_capture_and_on_two_streams():
    T, H = 1200, 2048
    xs = [rows_of_every_kind(T, H, torch.float16, 50 + i).cuda() for i in range(2)]
    plan = B.Plan(torch.float16, H, T, 6.0, [2, 4, 8], 0.2)
    refs = [R.encode(synth.raw_u16(x.cpu()), R.F16, 6.0, [2, 4, 8], 0.2) for x in xs]
    streams, bufs = [torch.cuda.Stream() for _ in range(2)], [plan.alloc(T) for _ in range(2)]
    torch.cuda.synchronize()
    for _ in range(20):
        for x, (blob, ws), s in zip(xs, bufs, streams):
            plan.encode(x, blob, ws, stream=s)
    torch.cuda.synchronize()
    for (blob, _), ref in zip(bufs, refs):
        assert_blobs_equal(blob.cpu().numpy(), ref)
    (blob, ws), x = bufs[0], xs[0].clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        plan.encode(x, blob, ws)
        plan.decode(blob, T, x, ws)
    x.copy_(xs[1])
    graph.replay()
    torch.cuda.synchronize()
    assert_blobs_equal(blob.cpu().numpy(), refs[1])
    assert np.array_equal(synth.raw_u16(x.cpu()), R.decode(refs[1]))


def test_workspace_initialised_for_fewer_rows():
    # large enough for the plan, cleared for a smaller one only: no row is written, and the status says so; calls within what was cleared, and calls
    # of one kernel, are not concerned
    H, bits = 256, [2, 4, 8]
    big, small = B.Plan(torch.float16, H, 3000, 6.0, bits, 0.2), B.Plan(torch.float16, H, 1400, 6.0, bits, 0.2)
    x = rows_of_every_kind(3000, H, torch.float16, 8)
    ws = torch.full((big.sizes(1)[1],), 0x11, dtype=torch.uint8, device="cuda")
    small.workspace_init(ws)
    for T in (1400, 100, 1399):
        check(big, x[:T], ws, bits)
    assert big.workspace_status(ws) == (0, 0)
    for T in (1401, 3000):
        blob = torch.full((big.sizes(T)[0],), 0xA5, dtype=torch.uint8, device="cuda")
        big.encode(x[:T].cuda(), blob, ws)
        assert big.blob_info(blob).status == 7 == big.workspace_status(ws)[0]
        lay = R.layout(H, T, 8, 0)
        assert (blob[lay["word_off"]:] == 0xA5).all()
        small.workspace_init(ws)
    big.workspace_init(ws)
    for T in (3000, 1400, 3000):
        check(big, x[:T], ws, bits)
    assert big.workspace_status(ws) == (0, 0)
