"""Parts of host-buffer calls with more rows than SMs: the one-kernel encoder with rows by ticket, which no other call takes."""
import time

import numpy as np
import pytest
import torch

from oracle import tsq_ref as R
from paper_2511_04002_b200 import binding as B

pytestmark = pytest.mark.gpu
TIMEOUT = 7
TICKET = 1                                                     # 32-bit word of the workspace's control block


def sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


class Call:
    """A host-buffer call's buffers, and the blob that it gives over a known fill."""

    def __init__(self, plan, x):
        self.plan, self.x, self.T = plan, x.pin_memory(), x.shape[0]
        self.blob, self.ws = plan.alloc(self.T)
        self.x_dev = torch.empty_like(x, device="cuda")
        self.host = torch.empty(self.blob.numel(), dtype=torch.uint8).pin_memory()

    def __call__(self):
        self.blob.fill_(0xA5)
        self.host.fill_(0xA5)
        torch.cuda.synchronize()
        try:
            self.plan.encode_host(self.x, self.host, self.x_dev, self.blob, self.ws)
        except B.TsqError as e:
            return e.status
        return 0

    def word(self, i, value=None):
        if value is not None:
            self.ws.view(torch.int32)[i] = value
        return int(self.ws.view(torch.int32)[i])


@pytest.mark.parametrize("hidden,part", [(8200, 445), (8200, 888), (4096, 593), (4096, 889)])
def test_a_part_without_its_first_row_leaves_the_next_ones_theirs(hidden, part):
    # the counter starts at 1: row 0 of the first part is never handed out, and that part runs out.  With 148 SMs 444 CTAs of the longer rows and 592 or 888 of the
    # shorter ones are resident: a part of one more has its last row among those and a CTA that has no number yet, which must not get one of the next part's
    T = 3 * part
    x = torch.randn((T, hidden), generator=torch.Generator().manual_seed(hidden)).to(torch.bfloat16)
    call = Call(B.Plan(torch.bfloat16, hidden, T, 6.0, [2, 4, 8], 0.2), x)
    assert call() == 0
    at = R.layout(hidden, T, 8, 0)["bits"]
    want = call.host.numpy()[at + part:at + T].copy()
    assert set(want) <= {2, 4, 8}
    for _ in range(20):
        call.plan.workspace_init(call.ws)
        call.plan.workspace_set_wait_limit(call.ws, 1000)
        call.word(TICKET, 1)
        assert call() == TIMEOUT and call.word(TICKET) == 0
        assert np.array_equal(call.blob[at + part:at + T].cpu().numpy(), want)
    call.plan.workspace_init(call.ws)
    assert call() == 0


def test_one_limit_for_a_part_of_two_turns():
    # the last row's CTA ends the call while other CTAs of the second turn have just started to poll: they must find that a wait has run out, not that the call
    # has ended, after which they would wait for a limit of their own
    part, hidden = 6 * sms(), 8200
    x = torch.randn((3 * part, hidden), generator=torch.Generator().manual_seed(1)).to(torch.bfloat16)
    call = Call(B.Plan(torch.bfloat16, hidden, 3 * part, 6.0, [2, 4, 8], 0.2), x)
    assert call() == 0
    ms = []
    for _ in range(24):
        call.plan.workspace_init(call.ws)
        call.plan.workspace_set_wait_limit(call.ws, 20000)
        call.word(TICKET, 1)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        assert call() == TIMEOUT
        ms.append(1e3 * (time.perf_counter() - t0))
    assert max(ms) < 1.5 * min(ms), ms                         # one limit, not two
