"""Calls of two kernels right behind one another: every call's number, slots, cells and input are its own, whatever the one before it has left.  Each call's
bytes are compared, of calls on a stream and of a graph's replays, with the input written by a kernel just before."""
import pytest
import torch

from paper_2511_04002_b200 import binding as B
from tests._parity import assert_blobs_equal
from tests.test_gpu_early_pack import reference
from tests.test_gpu_two_kernels import rows_of_every_kind

pytestmark = pytest.mark.gpu


def tensors(sizes, hidden, dtype, variant):
    xs = [rows_of_every_kind(T, hidden, dtype, 500 + i) for i, T in enumerate(sizes)]
    return [x.cuda() for x in xs], [reference(x, variant=variant) for x in xs]


@pytest.mark.parametrize("variant,hidden,sizes", [(0, 2048, (1500, 160, 1025)), (0, 4096, (200, 200, 149)), (0, 64, (4000, 2049, 33 * 32)),
                                                  (1, 2048, (300, 20, 31)), (1, 8200, (9, 150, 33))])
@pytest.mark.parametrize("captured", [False, True])
def test_every_call_behind_another(variant, hidden, sizes, captured):
    plan = B.Plan(torch.bfloat16, hidden, max(sizes), 6.0, [2, 4, 8], 0.2, variant=variant)
    ws = plan.alloc(1)[1]
    xd, refs = tensors(sizes, hidden, torch.bfloat16, variant)
    staged = torch.zeros_like(xd[0] if sizes[0] == max(sizes) else xd[sizes.index(max(sizes))])
    blobs = [[torch.full((plan.sizes(T)[0],), 0xA5, dtype=torch.uint8, device="cuda") for T in sizes] for _ in range(10)]
    out = [torch.empty_like(b) for b in blobs[0]]

    def calls(into):
        for x, blob, T in zip(xd, into, sizes):
            staged[:T].copy_(x)                                # what the call reads, by the kernel before it
            plan.encode(staged[:T], blob, ws)

    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        if captured:
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=stream):
                calls(out)
        for into in blobs:
            if captured:
                for o in out:
                    o.fill_(0xA5)
                graph.replay()
                for o, b in zip(out, into):
                    b.copy_(o)
            else:
                calls(into)
    torch.cuda.synchronize()
    assert plan.workspace_status(ws) == (0, 0)
    for into in blobs:
        for blob, ref in zip(into, refs):
            assert_blobs_equal(blob.cpu().numpy(), ref)
