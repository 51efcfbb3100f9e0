"""The conversions of the FP64 transforms in block floating point (fft_fx.cuh),
emulated in integers: FP64 bits -> integers under a common exponent -> FP64, and
the twiddle product with its rounding constant."""
import numpy as np
import pytest

M64 = (1 << 64) - 1


def bits(x):
    return int(np.float64(x).view(np.uint64))


def exponent(b):
    return (b >> 52) & 0x7FF


def from_bits(b, E, down):
    e, sh = exponent(b), E - exponent(b) + down
    m = ((b & 0xFFFFFFFFFFFFF) | (1 << 52)) << 8
    f = m >> sh if e != 0 and sh < 64 else 0
    return -f if b >> 63 else f


def to_double(f, X):
    u = abs(f)
    if u == 0:
        return 0.0
    n = 64 - u.bit_length()
    if 1023 + 63 - n + X < 1:
        return 0.0
    u = (u << n) & M64
    v, r = u >> 11, u & 0x7FF
    v += 1 if r > 0x400 or (r == 0x400 and v & 1) else 0
    v += (1023 + 63 - n + X - 1) << 52
    return float(np.uint64(v | ((1 << 63) if f < 0 else 0)).view(np.float64))


def s32(x):
    x &= 0xFFFFFFFF
    return x - (1 << 32) if x >> 31 else x


def split(x):
    return (x + 0x80000000) >> 32, s32(x)


def product(a, c):
    """Acc with one product: a c / 2^62."""
    (ah, al), (ch, cl) = split(a), split(c)
    mid = (1 << 29) + ah * cl + al * ch
    assert abs(mid) < 1 << 63 and abs(ah * ch) < 1 << 62
    return ((ah * ch) << 2) + (mid >> 30)


def test_round_trip_is_exact_near_the_largest_and_bounded_below_it():
    rng = np.random.default_rng(3)
    x = np.concatenate([rng.standard_normal(4000) * 10.0 ** rng.uniform(-12, 1, 4000), [0.0, 1.0, -1.0, 5e-324, 1e-308]])
    E = max(exponent(bits(v)) for v in x)
    unit = 2.0 ** (E - 1022 - 61)
    for v in x:
        f = from_bits(bits(v), E, 0)
        assert abs(f) < 1 << 61
        back = to_double(f, E - 1022 - 61)
        if E - exponent(bits(v)) <= 8:
            assert back == v  # all 53 bits fit
        assert abs(back - v) <= unit + abs(v) * 2.0 ** -53


def test_conversion_rounds_to_nearest_even_at_53_bits():
    for f, want in [((1 << 60) + 64, 1 << 60), ((1 << 60) + 128, 1 << 60), ((1 << 60) + 129, (1 << 60) + 256),
                    ((1 << 60) + 384, (1 << 60) + 512), ((1 << 61) - 1, 1 << 61), (-((1 << 61) - 1), -(1 << 61))]:
        assert to_double(f, 0) == float(want)


def test_twiddle_product_is_within_two_units_and_unbiased():
    rng = np.random.default_rng(4)
    err = []
    for _ in range(4000):
        a = int(rng.integers(-(1 << 61), 1 << 61))
        c = int(round(float(rng.uniform(-1, 1)) * 2.0 ** 62))
        num = a * c
        d = (product(a, c) << 62) - num  # in units of 2^-62
        err.append(d / 2.0 ** 62)
    err = np.array(err)
    # the rounding (1/2) and the dropped low x low part (up to 1)
    assert np.max(np.abs(err)) <= 1.5
    # zero mean: 4000 errors of at most 1.5 have a mean within 5 sigma of 0
    assert abs(np.mean(err)) <= 5 * 1.5 / np.sqrt(4000)
