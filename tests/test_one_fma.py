"""The scale of the 8-bit level and its codes by one FMA (divide_by, middle_up, one_fma_factor in csrc/tsq_encode_device.cuh), checked on
the CPU for every 16-bit maximum against the definition, clamp(rint(fl(m / s))) with s = fl(hi / 127); and what the sum of differences
without codes rests on: |(q >> 4) - low| is 0 or 1, and which it is follows from the 8-bit code but next to a step."""
import numpy as np
import pytest

f32 = np.float32


def patterns(fmt):
    if fmt == "f16":
        return np.arange(1, 0x7c00, dtype=np.uint16).view(np.float16).astype(f32)
    return (np.arange(1, 0x7f80, dtype=np.uint32) << 16).view(f32)


def fma(a, b, c):
    return (np.longdouble(a) * np.longdouble(b) + np.longdouble(c)).astype(f32)


@pytest.mark.parametrize("fmt", ["f16", "bf16"])
def test_scale_and_one_fma_codes_for_every_maximum(fmt):
    v = patterns(fmt)
    s = (v / f32(127)).astype(f32)
    ok = (s >= 2.0 ** -60) & (s <= 2.0 ** 60)
    inv = f32(1) / f32(127)
    q0 = (v * inv).astype(f32)
    quick = fma(fma(np.full_like(v, -127), q0, v), inv, q0)
    assert np.array_equal(quick[ok], s[ok])
    rem = fma(np.full_like(v, -127), s, v)
    half = (f32(0.5) * v).astype(f32)
    up = fma(np.full_like(v, -63.5), s, half) >= -f32(2.0 ** -19) * s
    assert np.array_equal(up[ok], ((half / s).astype(f32) >= f32(63.5))[ok])
    use = ok & (rem != 0)
    assert use.sum() > 0.98 * ok.sum()
    with np.errstate(over="ignore", divide="ignore", invalid="ignore"):
        r = (f32(1) / s).astype(f32)
    for ulp in (-1, 0, 1):                                   # the reciprocal may be one unit off
        factor = ((r.view(np.int32) + ulp).view(f32) * np.where(up, f32(1 + 2.0 ** -21), f32(1 - 2.0 ** -21))).astype(f32)
        for i in np.nonzero(use)[0][:: 1 if ulp == 0 else 17]:
            m = v[max(0, np.searchsorted(v, v[i] / 512)):i + 1]
            assert np.array_equal(np.rint((m / s[i]).astype(f32)), np.rint(m.astype(np.float64) * np.float64(factor[i]))), v[i]


def test_differences_are_at_most_one_and_lie_between_the_steps():
    rng = np.random.default_rng(0)
    for hi in np.concatenate([rng.uniform(0.5, 60000, 300), [1.0, 127.0, 254.0]]).astype(np.float16).astype(f32):
        m = patterns("f16")
        m = m[m <= hi]
        q = np.rint((m / f32(hi / f32(127))).astype(f32)).astype(int)
        low = np.rint((m / f32(hi / f32(7))).astype(f32)).astype(int)
        d = np.abs((q >> 4) - low)
        folded = np.minimum(q, 127 - q)
        j, n = folded >> 4, folded & 15
        assert d.max() <= 1
        assert (d[n > 9 + 2 * j] == 1).all() and (d[n < 9 + 2 * j] == 0).all()
