"""The codec's work as its users have it done, as timed cases.

A case is one call (or one encode + decode pair) on a [tokens x hidden] tensor of 16-bit activations, through the
public binding: Plan.encode / Plan.decode on device buffers, or Plan.encode_host / Plan.decode_host on pinned host
buffers.  Sizes and distributions are those of the repository's own workloads (synth.py, bench.py) and of its tests'
ragged shapes; the inputs are drawn on the GPU from the seed alone.

    listed()             the cases that stand for the range
    draw(rng)            one more case of the same range
    prepare(case, seed)  plan, buffers and inputs, as a program has them before the call
    run(state)           one pass through the public entry points
    work(case)           bytes and operations the pass cannot do without
    tolerance(case)      how far another correct implementation may be off
"""
from __future__ import annotations

import math
import random

import torch

from paper_2511_04002_b200 import binding as B

DELTA = 0.2                      # the distortion tolerance every workload of the repository uses
MAX_ELEMENTS = 32768 * 4096      # the largest tensor of the shape sweep
MAX_HOST_ELEMENTS = 4096 * 4096
BIT_SETS = {"2,4,8": (2, 4, 8), "2,3,4,8": (2, 3, 4, 8)}


def _case(op, tokens, hidden, dtype, base="normal", sigma=0.5, channels=0, gain=1.0, rate=0.0, tau=6.0, bits="2,4,8",
          signed=False, **name):
    """op: encode | decode | roundtrip (device buffers), host_roundtrip (pinned host buffers).  base: normal or
    student_t<nu>; sigma: spread of the per-token factor exp(N(0, sigma)); channels / gain: fixed outlier channels and
    their factor; rate: share of positions replaced by large values; signed: the signed-values variant."""
    return dict(name, op=op, tokens=tokens, hidden=hidden, dtype=dtype, base=base, sigma=sigma, channels=channels,
                gain=gain, rate=rate, tau=tau, bits=bits, signed=signed)


def listed():
    return [
        # one generated token leaves the device and comes back: launch and host latency, nothing else
        _case("roundtrip", 1, 4096, "f16", rate=0.001, name="token_roundtrip_1x4096_f16"),
        # a decode step of a batch of 64 sequences, each side of the link on its own machine
        _case("encode", 64, 4096, "f16", rate=0.001, name="step_encode_64x4096_f16"),
        _case("decode", 64, 4096, "f16", rate=0.001, name="step_decode_64x4096_f16"),
        # a short prompt, fixed outlier channels: the sender's side
        _case("encode", 128, 4096, "f16", channels=8, gain=50.0, name="prompt_encode_128x4096_f16"),
        # a 13B-shaped prefill with four candidate widths, each side
        _case("encode", 2048, 5120, "f16", "student_t4", channels=16, gain=30.0, bits="2,3,4,8", name="prefill_encode_2048x5120_f16"),
        _case("decode", 2048, 5120, "f16", "student_t4", channels=16, gain=30.0, bits="2,3,4,8", name="prefill_decode_2048x5120_f16"),
        # a 70B-shaped prefill, heavy tails, each side
        _case("encode", 8192, 8192, "bf16", "student_t3", sigma=0.0, rate=0.001, tau=8.0, name="prefill_encode_8192x8192_bf16"),
        _case("decode", 8192, 8192, "bf16", "student_t3", sigma=0.0, rate=0.001, tau=8.0, name="prefill_decode_8192x8192_bf16"),
        # the largest point of the shape sweep, one value in a hundred an outlier, both directions
        _case("roundtrip", 32768, 4096, "bf16", rate=0.01, name="bulk_roundtrip_32768x4096_bf16"),
        # a row length that is no multiple of a group or of a warp's work, an odd number of rows
        _case("roundtrip", 777, 3000, "bf16", rate=0.001, name="ragged_roundtrip_777x3000_bf16"),
        # the other reading of the quantiser (a plan option): codes of the signed values
        _case("roundtrip", 2048, 5120, "f16", "student_t4", channels=16, gain=30.0, bits="2,3,4,8", signed=True,
              name="signed_roundtrip_2048x5120_f16"),
        # a program that holds its tensors in pinned host memory: copies in, codec, copies out
        _case("host_roundtrip", 2048, 4096, "f16", rate=0.001, name="host_roundtrip_2048x4096_f16"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    op = rng.choice(["encode", "decode", "encode", "decode", "roundtrip", "host_roundtrip"])
    most = MAX_HOST_ELEMENTS if op == "host_roundtrip" else MAX_ELEMENTS
    hidden = 8 * _log_int(rng, 128, 2048) if rng.random() < 0.5 else rng.choice([2048, 4096, 5120, 6144, 8192, 12288, 16384])
    signed = rng.random() < 0.15
    if signed or hidden > 8192:
        most //= 2                               # these cost more per element
    tokens = min(_log_int(rng, 1, 32768), most // hidden)
    base, sigma = rng.choice([("normal", 0.5), ("student_t4", 0.5), ("student_t3", 0.0)])
    channels, gain, rate = rng.choice([(0, 1.0, 0.0), (0, 1.0, 0.001), (0, 1.0, 0.01), (8, 50.0, 0.0), (16, 30.0, 0.0)])
    return _case(op, tokens, hidden, rng.choice(["f16", "bf16"]), base, sigma, channels, gain, rate,
                 tau=8.0 if base == "student_t3" else 6.0, bits=rng.choice(sorted(BIT_SETS)), signed=signed)


def _dtype(case):
    return {"f16": torch.float16, "bf16": torch.bfloat16}[case["dtype"]]


def _activations(case, seed):
    """A hidden state of the case's distribution, on the GPU, from the seed alone."""
    T, H = case["tokens"], case["hidden"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.empty((T, H), dtype=_dtype(case), device="cuda")
    chan = torch.randperm(H, generator=g, device="cuda")[: case["channels"]]
    for t0 in range(0, T, 8192):
        n = min(T, t0 + 8192) - t0
        v = torch.randn((n, H), generator=g, device="cuda")
        if case["base"].startswith("student_t"):
            nu = int(case["base"][len("student_t"):])
            chi2 = sum(torch.randn((n, H), generator=g, device="cuda").square_() for _ in range(nu))
            v *= (chi2 / nu).rsqrt_()
        if case["sigma"] > 0:
            v *= torch.exp(torch.randn((n, 1), generator=g, device="cuda") * case["sigma"])
        v[:, chan] *= case["gain"]
        if case["rate"] > 0:
            hit = torch.rand((n, H), generator=g, device="cuda") < case["rate"]
            big = 40.0 + 10.0 * torch.randn((n, H), generator=g, device="cuda")
            v = torch.where(hit, torch.copysign(big, v), v)
        x[t0:t0 + n] = v.clamp_(-65504.0, 65504.0)
    return x


def _sections(blob, T, H, n_words):
    """Views of the blob's sections (the layout of include/tsq.h), planes and outlier list at their full capacity."""
    out, at = {"header": blob[:64]}, 64
    for name, n, dt in (("bits", T, torch.uint8), ("scale", T, torch.float32), ("zp", T, torch.int32),
                        ("word_off", T + 1, torch.int32), ("out_ptr", T + 1, torch.int32), ("words", n_words, torch.int32),
                        ("outl", T * H, torch.int32)):
        size = n * torch.empty(0, dtype=dt).element_size()
        out[name] = blob[at:at + size].view(dt)
        at += (size + 15) // 16 * 16
    return out


class State:
    pass


def prepare(case, seed):
    T, H, bits = case["tokens"], case["hidden"], BIT_SETS[case["bits"]]
    s = State()
    s.op, s.tokens = case["op"], T
    s.plan = B.Plan(_dtype(case), H, T, case["tau"], list(bits), DELTA, device=torch.cuda.current_device(),
                    variant=B.VARIANT_SIGNED_VALUES if case["signed"] else B.VARIANT_MAGNITUDES)
    s.x = _activations(case, seed)
    s.blob, s.ws = s.plan.alloc(T)
    s.blob.zero_()                               # what a call does not write stays zero
    s.y = torch.zeros_like(s.x)
    n_words = T * bits[-1] * ((H + 31) // 32)
    if s.op == "host_roundtrip":
        s.x_host = s.x.cpu().pin_memory()
        s.blob_host = torch.zeros(s.blob.numel(), dtype=torch.uint8).pin_memory()
        s.y_host = torch.zeros_like(s.x_host).pin_memory()
        s.out = {"blob": _sections(s.blob_host, T, H, n_words), "y": s.y_host}
        return s
    if s.op == "decode":
        s.plan.encode(s.x, s.blob, s.ws)         # what the sender sent
        s.out = {"y": s.y}
    elif s.op == "encode":
        s.out = {"blob": _sections(s.blob, T, H, n_words)}
    else:
        s.out = {"blob": _sections(s.blob, T, H, n_words), "y": s.y}
    return s


def run(s):
    if s.op == "host_roundtrip":
        s.plan.encode_host(s.x_host, s.blob_host, s.x, s.blob, s.ws)
        s.plan.decode_host(s.blob_host, s.tokens, s.y_host, s.blob, s.y, s.ws)
        return s.out
    if s.op != "decode":
        s.plan.encode(s.x, s.blob, s.ws)
    if s.op != "encode":
        s.plan.decode(s.blob, s.tokens, s.y, s.ws)
    return s.out


def work(case):
    """Tensor in and payload out for an encode, the mirror for a decode.  The payload: per-token fields, planes at the
    top candidate width (nearly every row keeps it) and one 4-byte entry per expected outlier.  Operations: threshold,
    minimum and maximum, quotient, rounding and code per element on the way in, product and rounding on the way out."""
    T, H = case["tokens"], case["hidden"]
    top = BIT_SETS[case["bits"]][-1]
    outliers = T * H * case["rate"] + T * case["channels"] * 0.9
    payload = 64 + 17 * T + T * ((H + 31) // 32) * 4 * top + 4 * outliers
    passes = 2 if case["op"] in ("roundtrip", "host_roundtrip") else 1
    return {"bytes": passes * (2 * T * H + payload), "flops": (6 if case["op"] != "decode" else 0) * T * H + (2 if case["op"] != "encode" else 0) * T * H}


def tolerance(case):
    """Codes, offsets and patterns are whole numbers, and the reconstruction is fixed to the bit by the format."""
    return "exact"
