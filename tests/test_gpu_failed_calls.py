"""What a two-kernel encode that fails leaves behind: the call behind one that does not fit its workspace.  (The failure is made on the host: a workspace
that was initialised for fewer rows.)"""
import pytest
import torch

from paper_2511_04002_b200 import binding as B
from tests._parity import assert_blobs_equal
from tests.test_gpu_early_pack import reference
from tests.test_gpu_two_kernels import rows_of_every_kind

pytestmark = pytest.mark.gpu
TIMEOUT = 7


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
