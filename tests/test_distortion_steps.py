"""The distortion sum that the encoders form without codes (add_differences, step_error in csrc/tsq_encode_device.cuh), restated in numpy
for every 16-bit magnitude of a row: with the corrections it is the sum over the true codes, without them it is never above it; and the
one-FMA codes of the levels of 2, 3 and 4 bits.  The reciprocal instruction's last bits are not known here: everything has to hold
for two units more and less in the factor (its error is below one, the product's half)."""
import numpy as np
import pytest

f32 = np.float32
MARGIN = 2.0 ** -19


def magnitudes(bits):
    """All significands of `bits` bits over twelve binades up to 1, as float64, ascending."""
    n = 1 << (bits - 1)
    m = np.arange(n, 2 * n) / n
    return np.unique(np.concatenate([m * 2.0 ** -e for e in range(1, 13)] + [[1.0]]))


def rn(x):
    return x.astype(np.float32).astype(np.float64)


def nudge(c, ulps):
    for _ in range(abs(ulps)):
        c = np.nextafter(c, f32(np.inf) if ulps > 0 else f32(0))
    return c


def true_difference(m, rng, b):
    code = np.rint((m.astype(f32) / (rng / f32(127))).astype(np.float64))
    low = np.rint((m.astype(f32) / (rng / f32((1 << (b - 1)) - 1))).astype(np.float64))
    return np.abs(np.floor(code / (1 << (8 - b))) - low)


def swept_difference(m, c, b):
    q = (1 << (b - 1)) - 1
    ratio = f32(127.0) / f32((1 << (8 - b)) * q)
    w = rn(m * np.float64(c) - 0.5 * q)                       # 11 + 24 bits and the constant: exact in binary64, rounded once
    ka, kb = np.float64(f32(ratio - f32(MARGIN) * ratio)), np.float64(f32(1.0 + MARGIN))
    return np.abs(np.floor(w * ka) - np.floor(w * kb))         # adding 1.5 * 2^23 rounding down: the floor of the exact product


def step_values(all_m, rng, b, dtype_bits):
    """The 16-bit magnitudes that step_error looks at."""
    q, sh = (1 << (b - 1)) - 1, 8 - b
    at = [k + 0.5 for k in range(q)] + [((j << sh) - 0.5) * q / 127 for j in range(1, q + 1) if 2 * j - 1 != q]
    at = np.array(at) / q * float(rng)
    near = all_m[np.clip(np.searchsorted(all_m, at), 1, len(all_m) - 1)]
    below = all_m[np.clip(np.searchsorted(all_m, at) - 1, 0, len(all_m) - 1)]
    near = np.where(np.abs(below - at) < np.abs(near - at), below, near)
    return near[np.abs(near - at) <= 2.0 ** -14 * at * (1 + 2.0 ** -20)]


@pytest.mark.parametrize("bits", [11, 8])
@pytest.mark.parametrize("b", [4, 3, 2])
def test_sum_is_exact_with_the_corrections_and_a_lower_bound_without(bits, b):
    grid, n = magnitudes(bits), 1 << (bits - 1)
    rng = np.random.default_rng(b)
    q = (1 << (b - 1)) - 1
    for sig in range(n, 2 * n):
        hi = sig / n
        all_m = np.concatenate([grid, np.arange(n, 2 * n) / n])
        # the smallest magnitude 0, as in every row with an outlier, or a 16-bit value up to hi / 256
        for lo in (0.0, rng.integers(n, 2 * n) / n * 2.0 ** -int(rng.integers(9, 12))):
            r = f32(hi) - f32(lo)
            m = np.concatenate([[0.0], all_m[(all_m <= hi) & (all_m >= lo)]])
            true = true_difference(m, r, b)
            near = step_values(all_m, r, b, bits)
            for ulps in (-2, 0, 2):
                c = nudge(f32(q) / r, ulps)
                swept = swept_difference(m, c, b)
                assert (swept <= true).all(), (hi, lo, ulps)
                off = m[swept != true]
                assert np.isin(off, near).all(), (hi, lo, ulps, off, near)


@pytest.mark.parametrize("bits", [11, 8])
@pytest.mark.parametrize("q,middle,half", [(127, 63.5, 2.0 ** -19), (7, 3.5, 2.0 ** -23), (3, 1.5, 2.0 ** -24), (1, 0.5, None)])
def test_scale_middle_and_one_fma_codes_of_a_level(bits, q, middle, half):
    n = 1 << (bits - 1)
    grid = magnitudes(bits)
    for sig in range(n, 2 * n):
        hi = f32(sig / n)
        s = hi / f32(q)
        if q > 1:                                              # divide_by: two roundings less than the division instruction
            inv = f32(1.0) / f32(q)
            q0 = hi * inv
            rem = f32(np.float64(hi) - q * np.float64(q0))
            assert f32(np.float64(q0) + np.float64(rem) * np.float64(inv)) == s
            tie = np.float64(hi) == q * np.float64(s)
            assert tie == (sig % q == 0)
        else:
            tie = False
        up = np.rint(np.float64((f32(0.5) * hi) / s)) > middle
        if half is not None:                                   # middle_up
            assert up == (0.5 * np.float64(hi) - middle * np.float64(s) >= -half * np.float64(s))
        else:
            assert not up                                      # 1/2 rounds to 0
        if tie:
            continue
        m = np.concatenate([[0.0], grid[grid <= hi], np.arange(n, sig + 1) / n])
        want = np.rint((m.astype(f32) / s).astype(np.float64))
        for ulps in (-1, 0, 1):
            r = nudge(f32(1.0) / s, ulps) * f32(1 + 2.0 ** -21 if up else 1 - 2.0 ** -21)
            for sign in (1.0, -1.0):                           # on the signed value, rounded as 1.5 * 2^23 + 128 + code
                got = np.rint(sign * m * np.float64(r))        # |m r| below 2^7 has its bits above 2^-53: exact enough to round
                assert (np.abs(got) == want).all(), (hi, ulps)
