"""Integer and double-float arithmetic that stands in for FP64-pipe instructions, replayed on the CPU operation
by operation: the rounding of kappa to float (fields.cu narrow), e^{-x} from the rate table and quotients by
a double-float reciprocal (march.cu exp_minus, quot_pos), and a source's twelfth (sources.cu twelfth).

Tolerances, from the operations: narrow and twelfth are exact roundings. exp_minus multiplies double-floats
good to about 2^-46 (a product drops its tails' product and rounds its error sum, at most 2^-44 each, three
of them): 2^-42 of e^{-x}. quot_pos corrects a quotient of a reciprocal within 2^-44 by its exact residual and
rounds once more: two units of 2^-53."""
import math
import os
import re
import struct
import sys
from fractions import Fraction

import numpy as np
import pytest

sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2512_12466_gb300", "csrc")


def bits(v):
    return struct.unpack("<Q", struct.pack("<d", v))[0]


def of_bits(b):
    return struct.unpack("<d", struct.pack("<Q", b))[0]


def narrow(v):
    b = bits(v)
    hi, lo = b >> 32, b & 0xffffffff
    u, rem = (((hi - 0x38000000) << 3) & 0xffffffff) | (lo >> 29), (lo << 3) & 0xffffffff
    if (hi - 0x38100000) & 0xffffffff >= 0x47f00000 - 0x38100000:
        if hi >= 0x47f00000:
            return 0x7fffffff if hi > 0x7ff00000 or (hi == 0x7ff00000 and lo) else 0x7f800000
        down = 897 - (hi >> 20)
        m = (((hi & 0xfffff) | 0x100000) << 32) | lo
        w = m >> down if down < 32 else 0
        sticky = down < 32 and (m & ((1 << down) - 1)) != 0
        u, rem = (w >> 29) & 0xffffffff, ((w << 3) & 0xffffffff) | int(sticky)
    return u + int(rem > 0x80000000 or (rem == 0x80000000 and u & 1))


@pytest.mark.parametrize("kind", ["normal", "subnormal", "ties", "ends"])
def test_narrow_rounds_as_the_conversion(kind):
    rng = np.random.default_rng(3)
    n = 20000
    if kind == "normal":
        v = np.exp(rng.uniform(-80, 80, n))
    elif kind == "subnormal":
        v = 2.0 ** rng.uniform(-180, -120, n)
    elif kind == "ties":                      # float midpoints, and their neighbours
        f = (2.0 ** rng.uniform(-148, 100, n)).astype(np.float32)
        mid = 0.5 * (f.astype(np.float64) + np.nextafter(f, np.float32(np.inf)).astype(np.float64))
        v = np.concatenate([mid, np.nextafter(mid, 0), np.nextafter(mid, np.inf)])
    else:
        v = np.array([0.0, 5e-324, 2.2e-308, 2.0 ** -150, 2.0 ** -149, np.nextafter(2.0 ** -150, 1), 2.0 ** -126,
                      np.nextafter(2.0 ** -126, 0), 3.4028234663852886e38, 3.4028235677973366e38, 1e39, 1e308, np.inf])
    with np.errstate(over="ignore", under="ignore"):
        want = v.astype(np.float32).view(np.uint32)
    assert [narrow(float(x)) for x in v] == want.tolist()


def rn(q):
    return float(q)                           # Fraction to float rounds to nearest, ties to even


def test_twelfth_is_the_rounded_quotient():
    rng = np.random.default_rng(4)
    y = 1.0 / 12.0
    for a in np.concatenate([np.exp(rng.uniform(-600, 600, 20000)), rng.integers(1, 1 << 53, 20000).astype(float)]):
        a = float(a)
        q = a * y
        assert rn(Fraction(q) + Fraction(rn(Fraction(a) - Fraction(q) * 12)) * Fraction(y)) == a / 12.0


@pytest.fixture(scope="module")
def rate():
    pytest.importorskip("mpmath")
    import test_rate_table as rt
    return rt


def test_exp_minus_table_and_value(rate):
    import mpmath as mp
    mp.mp.dps = 40
    src = open(os.path.join(CSRC, "march.cu")).read()
    body = src[src.index("kExpMinus2[kExpRows] = {"):]
    rows = re.findall(r"\{([-0-9.e+]+)f, ([-0-9.e+]+)f\}", body[:body.index("};")])
    rows = [(float(np.float32(h)), float(np.float32(l))) for h, l in rows]
    assert len(rows) == 28
    for m, (h, l) in enumerate(rows):
        assert abs((mp.mpf(h) + mp.mpf(l)) / mp.exp(-2 * m) - 1) < mp.mpf(2) ** -46
    tab = rate.header_rows()
    f32 = lambda v: float(np.float32(v))
    rng = np.random.default_rng(5)
    for x in np.concatenate([rng.uniform(2, 54, 1500), 2.0 * rng.integers(1, 27, 100), [2.0, 53.999999]]):
        x = float(x)
        h = of_bits(bits(x) & ~0x1fffffff)                        # df_of: the leading 24 bits and the rest
        l = f32(x - h)
        m = int(f32(0.5 * h))
        # r, then u = r g(r) and e = 1 - u as double-floats; their arithmetic is replayed by test_rate_table, so
        # g enters here as the double-float nearest to it
        rh, rl = Fraction(h) - 2 * m, Fraction(l)
        r = rh + rl
        g = float((1 - mp.exp(-mp.mpf(r.numerator) / r.denominator)) / (mp.mpf(r.numerator) / r.denominator)) if r else 1.0
        gh = f32(g)
        gl = f32(g - gh)
        r_h = f32(float(r))
        r_l = f32(float(r - Fraction(r_h)))

        def df_mul(a, b):
            p = rate.mul(a[0], b[0])
            e = rate.round32(Fraction(a[0]) * Fraction(b[0]) - Fraction(p))
            e = rate.round32(Fraction(a[0]) * Fraction(b[1]) + Fraction(e))
            return p, rate.round32(Fraction(a[1]) * Fraction(b[0]) + Fraction(e))

        u = df_mul((r_h, r_l), (gh, gl))
        s = rate.add(1.0, -u[0])
        err = float(Fraction(1) - Fraction(u[0]) - Fraction(s))   # two_sum's error is exact
        t = rate.add(err, rate.add(0.0, -u[1]))
        e0 = rate.add(s, t)
        e = (e0, float(Fraction(s) + Fraction(t) - Fraction(e0)))
        E = df_mul(e, rows[m])
        got = mp.mpf(E[0]) + mp.mpf(E[1])
        assert abs(got / mp.exp(-mp.mpf(x)) - 1) < mp.mpf(2) ** -42, x


def test_quot_pos_within_two_ulp():
    rng = np.random.default_rng(6)
    for _ in range(20000):
        a, b = float(np.exp(rng.uniform(-200, 200))), float(np.exp(rng.uniform(-200, 200)))
        e = math.frexp(b)[1] - 1
        bm = math.ldexp(b, -e)                                    # [1, 2)
        r = (1.0 / bm) * (1.0 + float(rng.uniform(-1, 1)) * 2.0 ** -44)
        q = a * r
        v = rn(Fraction(rn(Fraction(a) - Fraction(q) * Fraction(bm))) * Fraction(r) + Fraction(q))
        got = math.ldexp(v, -e)
        assert abs(Fraction(got) * Fraction(b) / Fraction(a) - 1) < Fraction(2, 1 << 53)
