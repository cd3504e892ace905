"""Parts of host-buffer calls with more rows than SMs: the one-kernel encoder with rows by ticket, which no other call takes."""
import time

import numpy as np
import pytest
import torch

from oracle import tsq_ref as R
from paper_2511_04002_b200 import binding as B
from paper_2511_04002_b200 import synth
from tests._parity import assert_blobs_equal
from tests.test_gpu_two_kernels import rows_of_every_kind

pytestmark = pytest.mark.gpu
TIMEOUT = 7
GEN, TICKET = 0, 1                                             # 32-bit words of the workspace's control block


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


def launches_of(call):
    before = B.kernel_launch_count()
    status = call()
    return status, B.kernel_launch_count() - before


def oracle(x, bits=(2, 4, 8), variant=0):
    return R.encode(synth.raw_u16(x), R.F16 if x.dtype == torch.float16 else R.BF16, 6.0, list(bits), 0.2, signed_values=variant == 1)


# rows of 5120 elements: an SM holds 3, 5 and 6 CTAs of the three register budgets, so 444, 740 and 888 rows at once on 148 SMs; rows of 40000: two groups per thread
@pytest.mark.parametrize("dtype,hidden,part", [(torch.float16, 5120, 420), (torch.float16, 5120, 600), (torch.bfloat16, 5120, 888), (torch.bfloat16, 1032, 888),
                                               (torch.float16, 16384, 160), (torch.bfloat16, 40000, 160)])
@pytest.mark.parametrize("bits", [(2, 4, 8), (2, 3, 6)])
def test_every_instance_by_ticket(dtype, hidden, part, bits):
    T = (3 if hidden > 1032 else 5) * part
    x = rows_of_every_kind(T, hidden, dtype, hidden + part)    # (some of them need the division instruction)
    call = Call(B.Plan(dtype, hidden, T, 6.0, list(bits), 0.2), x)
    assert launches_of(call) == (0, T // part)                 # one kernel per part
    assert_blobs_equal(call.host.numpy(), oracle(x, bits))
    assert call.plan.workspace_status(call.ws) == (0, 0) and call.word(TICKET) == 0


@pytest.mark.parametrize("hidden,parts", [(1024, 5), (4096, 3), (8200, 3)])  # sizes read in batches, one after another, by CTAs of more than 256 threads
def test_limits_of_a_few_polls_by_ticket(hidden, parts):
    T = parts * 6 * sms()
    x = rows_of_every_kind(T, hidden, torch.float16, hidden)
    ref = oracle(x)
    call = Call(B.Plan(torch.float16, hidden, T, 6.0, [2, 4, 8], 0.2), x)
    assert launches_of(call) == (0, parts)
    for k in range(24):
        call.plan.workspace_set_wait_limit(call.ws, 1 + (5 * k) % 32)
        status = call()
        assert status in (0, TIMEOUT)
        if status == 0:
            assert_blobs_equal(call.host.numpy(), ref)
            assert call.plan.workspace_status(call.ws) == (0, 0)
        else:
            assert call.plan.workspace_status(call.ws)[0] == TIMEOUT
            call.plan.workspace_init(call.ws)
    call.plan.workspace_set_wait_limit(call.ws, 0)
    assert call() == 0
    assert_blobs_equal(call.host.numpy(), ref)


LAST_GENERATION = (1 << 30) - 2                                # the part that runs as it wipes the rows' words, and the generations start over


@pytest.mark.parametrize("hidden,part", [(4096, 888), (8200, 300), (5120, 420)])
@pytest.mark.parametrize("before", [1, 2, 3])                  # the first, second or third part is the last of its generations
def test_generations_start_over_by_ticket(hidden, part, before):
    x = rows_of_every_kind(3 * part, hidden, torch.float16, 7)
    ref = oracle(x)
    call = Call(B.Plan(torch.float16, hidden, 3 * part, 6.0, [2, 4, 8], 0.2), x)
    torch.cuda.synchronize()
    call.word(GEN, LAST_GENERATION - before)
    for k in range(3):
        assert call() == 0
        assert_blobs_equal(call.host.numpy(), ref)
        assert call.word(GEN) == 3 * (k + 1) - before and call.word(TICKET) == 0
    assert call.plan.workspace_status(call.ws) == (0, 0)


@pytest.mark.parametrize("hidden,part", [(4096, 888), (8200, 888)])
def test_a_wait_that_runs_out_in_the_last_generation_by_ticket(hidden, part):
    x = rows_of_every_kind(3 * part, hidden, torch.float16, 8)
    call = Call(B.Plan(torch.float16, hidden, 3 * part, 6.0, [2, 4, 8], 0.2), x)
    call.plan.workspace_set_wait_limit(call.ws, 2000)
    torch.cuda.synchronize()
    call.word(GEN, LAST_GENERATION - 1)
    call.word(TICKET, 1)                                       # row 0 of the first part is never handed out
    assert call() == TIMEOUT
    assert call.word(GEN) == 2 and call.word(TICKET) == 0 and call.plan.workspace_status(call.ws)[0] == TIMEOUT
    call.plan.workspace_init(call.ws)
    assert call() == 0
    assert_blobs_equal(call.host.numpy(), oracle(x))


@pytest.mark.parametrize("dtype,variant,hidden", [(torch.float16, 0, 4096), (torch.float16, 1, 2048), (torch.bfloat16, 1, 4096)])
def test_both_sides_of_the_line_between_the_pack_shapes(dtype, variant, hidden):
    # rows of two and four segments of 1024 elements, of either kind of values; two kernels
    line = 120 * sms() // (hidden // 1024)
    few = rows_of_every_kind(500, hidden, dtype, hidden)
    x = few.repeat(line // 500 + 1, 1)[: line + 1].contiguous()
    ref, xd = oracle(x, variant=variant), x.cuda()
    plan = B.Plan(dtype, hidden, line + 1, 6.0, [2, 4, 8], 0.2, variant=variant)
    ws = plan.alloc(1)[1]
    for T in (line + 1, line):
        blob = torch.zeros(plan.sizes(T)[0], dtype=torch.uint8, device="cuda")
        plan.encode(xd[:T], blob, ws)
        got = blob.cpu().numpy()
        if T == line + 1:
            assert_blobs_equal(got, ref)
        else:                                                  # the rows before the last one are the same
            g, r = R.sections(got), R.sections(ref)
            for name in ("bits", "scale", "zp", "word_off", "out_ptr", "words", "outl"):
                assert np.array_equal(g[name], r[name][:g[name].size]), name
    assert plan.workspace_status(ws) == (0, 0)
