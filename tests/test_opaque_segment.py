"""The opaque segment of the FP64 table march (dtau >= 2), its device functions compiled for the host, against
40-digit arithmetic: e^{-x}, the photons absorbed, the budget left, and the quotient by a double-float reciprocal.

Tolerances, in units of u = 2^-53. exp_minus: its row of e^{-2m} (error computed here), u each from the rounding of
the middle factor's sum and of the product, and 2^-54 from the double-float e^{-r} - 1: the row and 2.5 u, 3 u
allowed. Absorbed: the error of e^{-x} times e^{-x} / (1 - e^{-x}) < 0.16, and two roundings of at most u / 2 above
0.86: 2 u. Left: e^{-x}'s, a rounding, and the tail of the double-float dropping 4 of 53 bits (2^-49): the row + 4 u +
2^-49. quot_pos: a reciprocal within 2^-44 corrected by the exact residual, and a rounding: u. The form with expm1,
which these operations replaced, left a budget good to (1.5 u e^x + 2^-49) at best; the new error stays below it.
Budgets are P m_G 2^64 with P from 1/12 down to 2^-30 (level 13) and m_G in [1, 2), so 2^34 to 2^61."""
import ctypes as C
import os
import re

import numpy as np
import pytest

from device_code import CSRC, compile_host, definition, source

mp = pytest.importorskip("mpmath")
U = 2.0 ** -53


@pytest.fixture(scope="module")
def dev(tmp_path_factory):
    df, m = source("dfloat.h"), source("march.cu")
    body = '#include "%s"\nusing namespace nyx;\n' % os.path.join(CSRC, "exp_table.h")
    body += "".join(definition(df, s) for s in ("struct dflt {", "__device__ __forceinline__ dflt df_two_sum(",
                                                "__device__ __forceinline__ dflt df_fast_two_sum(", "__device__ __forceinline__ dflt df_mul(",
                                                "__device__ __forceinline__ dflt df_add(", "__device__ __forceinline__ dflt df_rcp12(",
                                                "__device__ __forceinline__ dflt df_mant(", "__device__ __forceinline__ dflt df_of(",
                                                "__device__ __forceinline__ dflt df_of_near(",
                                                "__device__ __forceinline__ double widen_scaled(", "__device__ __forceinline__ double df_to_double("))
    body += re.search(r"constexpr int kExpRows = \d+;\n", m).group(0)
    body += "template <class R> struct Ieee { static bool lt(R a, R b) { return a < b; } };\n"
    body += "".join(definition(m, s) for s in ("__device__ constexpr float2 kExpMinus2[", "__device__ __forceinline__ double exp_minus(",
                                               "__device__ __forceinline__ double quot_pos(", "struct OpaqueSeg {",
                                               "__device__ __noinline__ OpaqueSeg opaque_segment("))
    lib = compile_host(tmp_path_factory.mktemp("opaque"), body + """
extern "C" double em(double x) { return exp_minus(x); }
extern "C" double quot(double a, double b) { return quot_pos(a, b); }
extern "C" void seg(double q, double dtau, double kap, double* out) {
    const dflt Q = df_of(q);
    const OpaqueSeg o = opaque_segment(Q, dtau, kap);
    out[0] = (double)Q.h + (double)Q.l; out[1] = o.aQ; out[2] = o.wd; out[3] = o.Q.h; out[4] = o.Q.l;
}
extern "C" void row(int m, double* out) { out[0] = kExpMinus2[m].x; out[1] = kExpMinus2[m].y; }
""")
    for f, n in ((lib.em, 1), (lib.quot, 2)):
        f.argtypes, f.restype = [C.c_double] * n, C.c_double
    lib.seg.argtypes = [C.c_double] * 3 + [C.c_void_p]
    mp.mp.dps = 40
    return lib


@pytest.fixture(scope="module")
def row_error(dev):
    out, err = np.empty(2), []
    for m in range(28):
        dev.row(m, out.ctypes.data_as(C.c_void_p))
        err.append(float(abs((mp.mpf(out[0]) + mp.mpf(out[1])) / mp.exp(-2 * m) - 1)))
    assert err[0] == 0.0 and err[1] < 2.0 ** -53 and max(err) < 2.0 ** -49
    return err


def depths():
    rng = np.random.default_rng(15)
    even = 2.0 * np.arange(1, 28)
    edge = np.concatenate([even, even + 1 / 512, np.arange(2 * 512 + 1, 8 * 512, 6) / 512])      # ends of rows and steps
    x = np.concatenate([rng.uniform(2, 4, 1500), rng.uniform(4, 8, 1000), rng.uniform(8, 55, 800), edge,
                        np.nextafter(edge, 0), np.nextafter(edge, 99)])
    return [float(v) for v in x if 2.0 <= v < 55.0]


def rel(got, want):
    return float(abs(got / want - 1))


def test_exp_minus(dev, row_error):
    for x in depths():
        m = int((x + 1 / 512) // 2)
        assert rel(mp.mpf(dev.em(x)), mp.exp(-mp.mpf(x))) <= row_error[m] + 3 * U, x
    for x in (57.0, 60.0, 63.99):
        assert 0.0 <= dev.em(x) < 2.0 ** -78


def test_segment(dev, row_error):
    rng = np.random.default_rng(16)
    out = np.empty(5)
    for x in depths():
        q, kap = float(np.exp(rng.uniform(24, 42))), float(np.exp(rng.uniform(-5, 5)))
        dev.seg(q, x, kap, out.ctypes.data)
        Q, e = mp.mpf(out[0]), mp.exp(-mp.mpf(x))
        assert rel(mp.mpf(out[1]), Q * (1 - e)) <= 2 * U, x
        assert rel(mp.mpf(out[2]) * mp.mpf(kap), mp.mpf(out[1])) <= 1.01 * U, x
        left = rel(mp.mpf(out[3]) + mp.mpf(out[4]), Q * e)
        m = int((x + 1 / 512) // 2)
        assert left <= row_error[m] + 4 * U + 2.0 ** -49, x
        assert left <= 1.5 * U * np.exp(x) + 2.0 ** -49, x
    dev.seg(3.0, 80.0, 2.0, out.ctypes.data)
    assert out[1] == 3.0 and out[2] == 1.5 and out[3] == 0.0 and out[4] == 0.0


def test_quotient(dev):
    rng = np.random.default_rng(17)
    for _ in range(20000):
        a, b = float(np.exp(rng.uniform(-200, 200))), float(np.exp(rng.uniform(-200, 200)))
        assert rel(mp.mpf(dev.quot(a, b)) * mp.mpf(b), mp.mpf(a)) <= 1.01 * U, (a, b)
    for a, b in ((1.0, 5e-324), (0.0, 3.0), (1e-300, 1e300), (1e300, 1e-300), (5.0, np.inf)):
        with np.errstate(over="ignore", under="ignore"):
            assert dev.quot(a, b) == float(np.float64(a) / np.float64(b)), (a, b)
