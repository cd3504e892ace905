"""The distortion sum of signed-values rows in which a code needs the clamp, as sizes_kernel in csrc/tsq_encode.cu forms it, restated in
numpy: codes unclamped and modulo 256, then the largest value's share exchanged for the true one.  Checked against the definition,
|(clamp(top code) >> shift) - clamp(lower code)|; that only the largest value's code can need the clamp is checked as well."""
import numpy as np
import pytest

from oracle import tsq_ref as R

f32 = np.float32


def values(fmt, below=6.0):
    """Every 16-bit value of magnitude under `below`, ascending, as binary32."""
    p = np.arange(0x10000, dtype=np.uint32)
    v = p.astype(np.uint16).view(np.float16).astype(f32) if fmt == "f16" else (p << 16).view(f32)
    return np.unique(v[np.abs(v) < below])


def level(lo, hi, b):
    """(scale, zero-point, Q_max) as Eq. "Proposed" has them on the signed values."""
    q = (1 << b) - 1
    s = (hi - lo) / f32(q) if hi > lo else (abs(hi) if hi != 0 else f32(1))
    return s, int(np.rint(lo / s)), q


def codes(m, lv):
    return np.rint((m / lv[0]).astype(f32)).astype(np.int64) - lv[1]


def true_sum(m, count, top, low, sh):
    d = np.abs((np.clip(codes(m, top), 0, top[2]) >> sh) - np.clip(codes(m, low), 0, low[2]))
    return int((d * count).sum())


def packed_sum(m, count, top, low, sh):
    """Without clamps: the codes' low bytes."""
    return int((np.abs(((codes(m, top) & 255) >> sh) - (codes(m, low) & 255)) * count).sum())


def exchanged(s, hi, n_largest, top, low, sh):
    code, lower = int(codes(np.array([hi], f32), top)[0]), int(codes(np.array([hi], f32), low)[0])
    return s + n_largest * (abs((min(code, top[2]) >> sh) - min(lower, low[2])) - abs(((code & 255) >> sh) - (lower & 255)))


PAIRS = [(8, 4), (8, 3), (8, 2), (6, 3), (5, 2), (3, 2)]


@pytest.mark.parametrize("fmt", ["f16", "bf16"])
def test_sum_of_symmetric_rows(fmt):
    v = values(fmt)
    ones = 0
    for hi in v[v >= 2.0 ** -7]:
        m, count = np.array([-hi, hi], f32), np.array([3096, 1000])
        for bt, bl in PAIRS:
            top, low = level(-hi, hi, bt), level(-hi, hi, bl)
            want = true_sum(m, count, top, low, bt - bl)
            assert exchanged(packed_sum(m, count, top, low, bt - bl), hi, 1000, top, low, bt - bl) == want, (hi, bt, bl)
            ones += true_sum(m[1:], count[1:], top, low, bt - bl) != 0
    assert ones > 0                                            # the largest value's difference is not always 0


@pytest.mark.parametrize("fmt", ["f16", "bf16"])
def test_only_the_largest_value_needs_the_clamp(fmt):
    v = values(fmt)
    rng = np.random.default_rng(5)
    clamped = 0
    for k in range(400):
        hi = rng.choice(v[v > 2.0 ** -10])
        lo = (-hi, rng.choice(v[v < hi]), -hi / 2, f32(0))[k % 4] if k % 16 else -rng.choice(v[(v > hi) & (v < 300 * hi)])
        m = v[(v >= lo) & (v <= hi)]
        if not m.size or m[0] != lo or lo == hi:
            continue
        count = rng.integers(1, 50, m.size)
        for bt, bl in PAIRS:
            top, low = level(lo, hi, bt), level(lo, hi, bl)
            for lv in (top, low):
                c = codes(m, lv)
                assert c[0] == 0 and c.min() >= 0 and (c[:-1] <= lv[2]).all() and c[-1] <= lv[2] + 1
                clamped += c[-1] > lv[2]
            got = exchanged(packed_sum(m, count, top, low, bt - bl), hi, int(count[-1]), top, low, bt - bl)
            assert got == true_sum(m, count, top, low, bt - bl), (lo, hi, bt, bl)
    assert clamped > 50


def test_widths_of_saturated_rows():
    """Rows of +v and -v whose lower candidate fails only by the largest value's differences: the sum decides as the oracle does."""
    v = 0.011474609375
    row = np.full((1, 4096), np.array([-v], f32).view(np.uint32)[0] >> 16, np.uint16)
    row[:, :1000] = np.array([v], f32).view(np.uint32)[0] >> 16
    for bits in ([4, 8], [2, 4, 8], [2, 3, 4, 8]):
        blob = R.encode(row, R.BF16, 6.0, bits, 0.2, signed_values=True)
        assert R.sections(blob)["bits"].tolist() == [8]
        top, low = level(f32(-v), f32(v), 8), level(f32(-v), f32(v), bits[-2])
        m, count = np.array([-v, v], f32), np.array([3096, 1000])
        assert exchanged(packed_sum(m, count, top, low, 8 - bits[-2]), f32(v), 1000, top, low, 8 - bits[-2]) > int(0.2 * 4096)
