"""The second kernel of a two-kernel encode starts while the first still runs: rows that are sized late in front of rows that are packed early, calls one after
another on one workspace with the numbers of calls starting over, blocks of 32, 1024 and 32768 rows that end with the call, and the shapes of the second
kernel on both sides of their line."""
import pytest
import torch

from oracle import tsq_ref as R
from paper_2511_04002_b200 import binding as B
from paper_2511_04002_b200 import synth
from tests._parity import assert_blobs_equal
from tests.test_gpu_two_kernels import rows_of_every_kind

pytestmark = pytest.mark.gpu
LAST_CALL = (1 << 30) - 2                                      # the call that wipes the slots as it ends
CALLS_WORD = 9                                                 # where the workspace counts calls of two kernels


def reference(x, bits=(2, 4, 8), variant=0):
    code = R.F16 if x.dtype == torch.float16 else R.BF16
    return R.encode(synth.raw_u16(x), code, 6.0, list(bits), 0.2, signed_values=variant == 1)


@pytest.mark.parametrize("tokens,hidden", [(149, 1024), (151, 4096), (160, 8200), (2049, 64), (32769, 16)])
def test_numbers_of_calls_start_over(tokens, hidden):
    plan = B.Plan(torch.float16, hidden, tokens, 6.0, [2, 4, 8], 0.2)
    ws = plan.alloc(1)[1]
    x = rows_of_every_kind(tokens, hidden, torch.float16, tokens)
    ref, xd = reference(x), x.cuda()
    torch.cuda.synchronize()
    ws.view(torch.int32)[CALLS_WORD] = LAST_CALL - 3
    for k in range(6):
        blob = torch.full((plan.sizes(tokens)[0],), 0xA5, dtype=torch.uint8, device="cuda")
        plan.encode(xd, blob, ws)
        assert_blobs_equal(blob.cpu().numpy(), ref)
    assert plan.workspace_status(ws) == (0, 0) and int(ws.view(torch.int32)[CALLS_WORD]) == 3


@pytest.mark.parametrize("variant", [0, 1])
def test_calls_one_after_another_with_other_inputs(variant):
    # no call may take a slot or a cell of the one before it for its own: other tensors, other sizes, no wait between the calls
    H, sizes = 2048, (1500, 149, 1024, 1500, 200, 1025, 33 * 32, 1499)
    plan = B.Plan(torch.bfloat16, H, 1500, 6.0, [2, 4, 8], 0.2, variant=variant)
    ws = plan.alloc(1)[1]
    xs = [rows_of_every_kind(T, H, torch.bfloat16, 70 + i) for i, T in enumerate(sizes)]
    xd = [x.cuda() for x in xs]
    blobs = [torch.zeros(plan.sizes(T)[0], dtype=torch.uint8, device="cuda") for T in sizes]
    torch.cuda.synchronize()
    for _ in range(3):
        for x, blob in zip(xd, blobs):
            plan.encode(x, blob, ws)
    torch.cuda.synchronize()
    assert plan.workspace_status(ws) == (0, 0)
    for x, blob in zip(xs, blobs):
        assert_blobs_equal(blob.cpu().numpy(), reference(x, variant=variant))


@pytest.mark.parametrize("hidden", [2048, 3072, 4096])
def test_both_sides_of_the_line_between_the_pack_shapes(hidden):
    segments = hidden // 1024
    line = 120 * torch.cuda.get_device_properties(0).multi_processor_count // segments
    plan = B.Plan(torch.bfloat16, hidden, line + 1, 6.0, [2, 4, 8], 0.2)
    ws = plan.alloc(1)[1]
    few = rows_of_every_kind(500, hidden, torch.bfloat16, hidden)
    x = few.repeat((line + 500) // 500, 1)[: line + 1].contiguous()
    ref = reference(x[: line + 1])
    blob = torch.zeros(plan.sizes(line + 1)[0], dtype=torch.uint8, device="cuda")
    plan.encode(x.cuda(), blob, ws)
    assert_blobs_equal(blob.cpu().numpy(), ref)
    blob = torch.zeros(plan.sizes(line)[0], dtype=torch.uint8, device="cuda")
    plan.encode(x[:line].cuda(), blob, ws)
    assert_blobs_equal(blob.cpu().numpy(), reference(x[:line]))


@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16])
@pytest.mark.parametrize("variant", [0, 1])
def test_subnormal_values(dtype, variant):
    # values are widened by an addition: exact for subnormal ones as well
    T, H = 300, 1032
    g = torch.Generator().manual_seed(5)
    raw = torch.randint(0, 1 << (10 if dtype == torch.float16 else 7), (T, H), generator=g).to(torch.int16)
    x = (raw | (torch.randint(0, 2, (T, H), generator=g) << 15).to(torch.int16)).view(dtype).contiguous()
    plan = B.Plan(dtype, H, T, 6.0, [2, 4, 8], 0.2, variant=variant)
    blob, ws = plan.alloc(T)
    blob.zero_()
    plan.encode(x.cuda(), blob, ws)
    assert_blobs_equal(blob.cpu().numpy(), reference(x, variant=variant))
