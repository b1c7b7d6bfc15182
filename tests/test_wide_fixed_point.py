"""The 64-bit form's fixed-point quantiser (csrc/gpz_wide_fast.cu: wide_code) in
Python integers: wherever it does not ask for fp64, its code is the format's
first candidate floor(RN(fma(RN(x - min), inv, 1/2))), computed exactly --
random and adversarial values (on and next to the half steps) over steps of
many magnitudes, ranges of up to 2^40 steps and offsets of up to 2^45 bounds."""
import random
from fractions import Fraction

import pytest


def rn(q):
    """The double nearest to a rational (ties to even: float() of a Fraction)."""
    return float(q)


def fixed(x, rs):
    m, e = abs(x), 0
    import struct
    bits = struct.unpack("<Q", struct.pack("<d", m))[0]
    e = bits >> 52
    v = (((bits & ((1 << 52) - 1)) | (1 << 52)) << 10) & ((1 << 64) - 1)
    sh = (rs - e) & 0xffffffff
    v = 0 if sh > 63 else v >> sh
    return -v if x < 0 else v


def code(x, mn, s, inv):
    """(code, certain) as the kernel computes them."""
    import math
    es = math.frexp(s)[1] - 1
    k = es - 15
    rs = 1085 + k
    d = fixed(x, rs) - fixed(mn, rs)
    assert 0 <= d < 1 << 64
    m = Fraction(inv) * Fraction(2) ** (k + 78)
    assert m.denominator == 1 and 1 << 62 <= m <= 1 << 63
    m = int(m)
    dl, dh, ml, mh = d & 0xffffffff, d >> 32, m & 0xffffffff, m >> 32
    t = dh * mh + ((dl * mh) >> 32) + 8192 + ((dh * ml) >> 32)
    assert t < 1 << 64
    return t >> 14, ((t + 10) & 16383) >= 20


@pytest.mark.parametrize("exp", [-990, -300, -30, -1, 0, 1, 40, 700])
@pytest.mark.parametrize("log_range", [0, 8, 20, 33, 40])
def test_certain_codes_are_first_candidates(exp, log_range):
    rng = random.Random(exp * 100 + log_range)
    certain = 0
    for trial in range(300):
        eb = rng.uniform(1.0, 2.0) * 2.0 ** exp
        if trial % 7 == 0:
            eb = 2.0 ** exp * (64.0 / 63.0 if trial % 2 else 1.0)  # steps at and next to powers of two
        s = eb * 1.96875
        inv = 1.0 / s
        off = rng.choice([0.0, 1.0, -1.0]) * eb * 2.0 ** rng.uniform(0, 44.9)
        q = rng.randrange(0, 1 << log_range) if log_range else 0
        frac = rng.choice([0.0, 0.5, 0.49999999, 0.50000001, rng.random(), 2.0 ** -13, 1 - 2.0 ** -14])
        mn = off
        x = rn(Fraction(mn) + (q + Fraction(frac)) * Fraction(s))
        if x < mn or abs(x) > eb * 2.0 ** 45 or x - mn > s * 2.0 ** 40:
            continue
        t = rn(Fraction(rn(Fraction(x) - Fraction(mn))) * Fraction(inv) + Fraction(1, 2))
        got, sure = code(x, mn, s, inv)
        if sure:
            certain += 1
            assert got == int(t), (x, mn, s)
    assert certain > 60
