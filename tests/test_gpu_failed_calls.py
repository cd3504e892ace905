"""What a two-kernel encode that fails leaves behind, and how it ends: the call behind one that does not fit its workspace, and rows whose place never
comes.  The failures are made on the host: a workspace that was initialised for fewer rows, a count in the workspace that cannot come out."""
import pytest
import torch

from paper_2511_04002_b200 import binding as B
from tests._parity import assert_blobs_equal
from tests.test_gpu_early_pack import reference
from tests.test_gpu_two_kernels import rows_of_every_kind

pytestmark = pytest.mark.gpu
OK, TIMEOUT = 0, 7


@pytest.mark.parametrize("before", [0, 1])                     # calls before the first one that fails: odd and even numbers
@pytest.mark.parametrize("variant,fits,hidden", [(0, 200, 4096), (0, 1400, 2048), (0, 33 * 32, 1024), (1, 20, 8192), (1, 300, 2048)])
def test_a_call_behind_one_that_does_not_fit(variant, fits, hidden, before):
    # the second kernel of the call that fits starts while its first still runs: it must not take what the failed call has left for its own
    more = 3 * fits
    big = B.Plan(torch.bfloat16, hidden, more, 6.0, [2, 4, 8], 0.2, variant=variant)
    small = B.Plan(torch.bfloat16, hidden, fits, 6.0, [2, 4, 8], 0.2, variant=variant)
    ws = torch.zeros(big.sizes(1)[1], dtype=torch.uint8, device="cuda")
    small.workspace_init(ws)
    xs = [rows_of_every_kind(fits, hidden, torch.bfloat16, 300 + i) for i in range(3)]
    refs = [reference(x, variant=variant) for x in xs]
    xd = [x.cuda() for x in xs]
    fails = rows_of_every_kind(more, hidden, torch.bfloat16, 299).cuda()
    for _ in range(before):
        big.encode(xd[0], torch.zeros(big.sizes(fits)[0], dtype=torch.uint8, device="cuda"), ws)
    calls = []
    torch.cuda.synchronize()
    for k in range(12):
        for T, x in ((more, fails), (fits, xd[k % 3]), (fits, xd[(k + 1) % 3]))[: 2 + k % 2]:
            calls.append((T, torch.full((big.sizes(T)[0],), 0xA5, dtype=torch.uint8, device="cuda"), k, x))
    torch.cuda.synchronize()
    for T, blob, k, x in calls:
        big.encode(x, blob, ws)
    torch.cuda.synchronize()
    for T, blob, k, x in calls:
        if T == more:
            assert big.blob_info(blob).status == TIMEOUT
        else:
            assert_blobs_equal(blob.cpu().numpy(), refs[[x.data_ptr() for x in xd].index(x.data_ptr())])
    assert big.workspace_status(ws)[0] == TIMEOUT


BLOCKS_AT, BLOCK_WORDS, CELLS = 2 * 2048 + 8, 80, {32: 64, 1024: 66, 32768: 68}  # 64-bit words behind the control block of 8
CALLS_WORD = 9                                                 # 32-bit word of the control block: calls of two kernels that have ended


@pytest.mark.parametrize("tokens,hidden,block,row", [(300, 4096, 32, 64),       # the last row among those without a place
                                                     (2100, 512, 32, 64),       # the last row has its place: its block of 1024 is whole
                                                     (2100, 512, 1024, 0),
                                                     (66000, 16, 32768, 0), (66000, 16, 1024, 1024)])
@pytest.mark.parametrize("limit", [0, 3000])
def test_a_count_that_never_comes_out(tokens, hidden, block, row, limit):
    plan = B.Plan(torch.float16, hidden, tokens, 6.0, [2, 4, 8], 0.2)
    ws = plan.alloc(1)[1]
    x = rows_of_every_kind(tokens, hidden, torch.float16, tokens)
    ref, xd = reference(x), x.cuda()
    blob = torch.full((plan.sizes(tokens)[0],), 0xA5, dtype=torch.uint8, device="cuda")
    plan.encode(xd, blob, ws)
    for parity in range(2):
        plan.workspace_set_wait_limit(ws, limit)
        turn = (int(ws.view(torch.int32)[CALLS_WORD]) + 1) & 1
        ws.view(torch.int64)[8 + BLOCKS_AT + BLOCK_WORDS * (row // 32) + CELLS[block] + turn] = 1 << 51  # one row (or block) too many
        blob.fill_(0xA5)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        e0.record()
        plan.encode(xd, blob, ws)
        e1.record()
        torch.cuda.synchronize()
        assert plan.blob_info(blob).status == TIMEOUT and plan.workspace_status(ws)[0] == TIMEOUT
        # the first kernel takes under 0.2 ms, and each of 30 turns of CTAs 64 polls of 3 us at most
        assert e0.elapsed_time(e1) < 20.0
        plan.workspace_init(ws)
        for _ in range(1 + parity):
            blob.fill_(0xA5)
            plan.encode(xd, blob, ws)
            assert_blobs_equal(blob.cpu().numpy(), ref)
        assert plan.workspace_status(ws) == (OK, OK)
