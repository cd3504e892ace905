"""The decoder on blobs put together row by row: every bit-width next to every other (so that plane words start at any 4-byte boundary), scales and
zero-points on both sides of the fused form, lists of outliers from none to a whole row, at the row counts where the kernel instance changes."""
import numpy as np
import pytest
import torch

from oracle import tsq_ref as R
from paper_2511_04002_b200 import binding as B
from tests._parity import gpu_decode

pytestmark = pytest.mark.gpu
BITS = [2, 3, 4, 5, 6, 7, 8]


def blob_of_any_rows(tokens, hidden, dtype, signed, seed):
    rng = np.random.default_rng(seed)
    lay, wpp = R.layout(hidden, tokens, 8, 0), (hidden + 31) // 32
    blob = np.zeros(R.encode(np.zeros((tokens, hidden), np.uint16), dtype, 6.0, BITS, 0.2, signed_values=signed).size, np.uint8)
    blob[:64] = R.encode(np.zeros((tokens, hidden), np.uint16), dtype, 6.0, BITS, 0.2, signed_values=signed)[:64]

    def put(name, a):
        blob[lay[name]:lay[name] + a.nbytes] = np.ascontiguousarray(a).view(np.uint8)

    b = rng.integers(2, 9, tokens)
    scale = rng.choice([2.0 ** -140, 2.0 ** -20, 0.0123, 0.37, 1.0, 2.0 ** 15, 2.0 ** 99, 2.0 ** 100, 2.0 ** 101, 2.0 ** 120], tokens)
    least = 1 - 2 ** 22 if signed else 0
    zp = np.where(rng.random(tokens) < 0.5, 0, rng.choice([1, 77, 2 ** 22 - 1, least, least // 3], tokens))
    count = np.minimum(hidden, rng.choice([0, 0, 1, 3, 33, 300, 600, hidden], tokens, p=[.2, .2, .2, .1, .1, .1, .05, .05]))
    word_off = np.concatenate([[0], np.cumsum(b * wpp)])
    out_ptr = np.concatenate([[0], np.cumsum(count)])
    words = rng.integers(0, 2 ** 32, word_off[-1], dtype=np.uint32)
    cols = np.concatenate([np.sort(rng.permutation(hidden)[:n]) for n in count]).astype(np.uint32)
    put("bits", b.astype(np.uint8))
    put("scale", scale.astype(np.float32))
    put("zp", zp.astype(np.int32))
    put("word_off", word_off.astype(np.uint32))
    put("out_ptr", out_ptr.astype(np.uint32))
    put("words", words)
    put("outl", cols << 16 | rng.integers(0, 2 ** 16, cols.size, dtype=np.uint32))
    blob[40:48] = np.array([word_off[-1]], np.uint64).view(np.uint8)
    blob[48:56] = np.array([out_ptr[-1]], np.uint64).view(np.uint8)
    y = R.decode(blob)
    row = np.repeat(np.arange(tokens), count)
    y[row, cols] = blob[lay["outl"]:lay["outl"] + 4 * cols.size].view(np.uint32) & 0xffff   # an outlier's slot holds the outlier
    return blob, y


@pytest.mark.parametrize("signed", [False, True])
@pytest.mark.parametrize("threads_per_sm", [0, 1059, 1062, 2559, 2562])
@pytest.mark.parametrize("dtype,hidden", [(torch.float16, 8), (torch.bfloat16, 1000), (torch.float16, 5120), (torch.bfloat16, 16384),
                                          (torch.float16, 16392)])
def test_rows_of_every_width(dtype, hidden, threads_per_sm, signed):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    threads = min(512, (hidden + 1023) // 1024 * 32)
    tokens = max(5, threads_per_sm * sms // threads)
    blob, want = blob_of_any_rows(tokens, hidden, R.F16 if dtype == torch.float16 else R.BF16, signed, hidden + threads_per_sm)
    plan = B.Plan(dtype, hidden, tokens, 6.0, BITS, 0.2, variant=B.VARIANT_SIGNED_VALUES if signed else B.VARIANT_MAGNITUDES)
    ws = plan.alloc(1)[1]
    got = gpu_decode(plan, torch.from_numpy(blob).cuda(), tokens, ws)
    assert np.array_equal(got, want), np.argwhere(got != want)[:4]
    assert plan.workspace_status(ws) == (0, 0)


@pytest.mark.parametrize("hidden", [1000, 4096])
def test_first_outliers_of_long_calls_in_turn(hidden):
    # The 32-register instance, whose threads take their first outlier through shared memory: two blobs with other lists in turn, so that
    # an entry read too early is one of the other blob's.
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    tokens = 2562 * sms // ((hidden + 1023) // 1024 * 32)
    blobs = [blob_of_any_rows(tokens, hidden, R.F16, False, hidden + k) for k in range(2)]
    plan = B.Plan(torch.float16, hidden, tokens, 6.0, BITS, 0.2)
    ws = plan.alloc(1)[1]
    on_device = [torch.from_numpy(blob).cuda() for blob, _ in blobs]
    want = [torch.from_numpy(y.view(np.int16)).cuda() for _, y in blobs]
    y = torch.empty((tokens, hidden), dtype=torch.float16, device="cuda")
    for k in range(40):
        plan.decode(on_device[k % 2], tokens, y, ws)
        assert torch.equal(y.view(torch.int16), want[k % 2]), "call %d" % k
    assert plan.workspace_status(ws) == (0, 0)
