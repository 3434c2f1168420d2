"""The optical depth as the per-cell pass stores it: k where the cell may receive a secondary deposit, -k
elsewhere, in FP32 rounded to the nearest float. A -0.0 in n_H (valid input) makes k negative zero."""
import ctypes as C

import numpy as np
import pytest

from device_code import compile_host, definition, source


@pytest.fixture(scope="module")
def dev(tmp_path_factory):
    src = source("fields.cu")
    body = "".join(definition(src, s) for s in ("__device__ __forceinline__ long long bits_of(",
                                                "__device__ __forceinline__ float narrow(",
                                                "__device__ __forceinline__ R stored_kappa(",
                                                "inline double ordered_threshold(",
                                                "__device__ __forceinline__ bool eligible("))
    return compile_host(tmp_path_factory.mktemp("kappa"), body + """
extern "C" void f32(const double* k, int n, int elig, float* out) { for (int i = 0; i < n; ++i) out[i] = stored_kappa<float>(k[i], elig); }
extern "C" void f64(const double* k, int n, int elig, double* out) { for (int i = 0; i < n; ++i) out[i] = stored_kappa<double>(k[i], elig); }
extern "C" int elig(double nh, double x, double n_th) { return eligible(nh, (1.0 - x) * nh, ordered_threshold(n_th)); }
""")


def run(dev, name, dtype, k, elig):
    out = np.empty(len(k), dtype=dtype)
    getattr(dev, name)(k.ctypes.data_as(C.c_void_p), len(k), elig, out.ctypes.data_as(C.c_void_p))
    return out


@pytest.mark.parametrize("elig", [0, 1])
def test_stored_kappa_is_the_rounded_signed_value(dev, elig):
    rng = np.random.default_rng(8)
    k = np.concatenate([[0.0, 5e-324, 2.0 ** -150, 2.0 ** -149, 2.0 ** -126, 2.2e-16, 3.4028235677973366e38, 1e39, np.inf],
                        np.exp(rng.uniform(-110, 88, 5000)), 2.0 ** rng.uniform(-160, -120, 2000)])
    k = np.concatenate([k, -k])
    assert np.signbit(k[len(k) // 2]) and k[len(k) // 2] == 0.0
    want = k if elig else -k
    with np.errstate(over="ignore", under="ignore"):
        want32 = want.astype(np.float32)
    assert np.array_equal(run(dev, "f32", np.float32, k, elig).view(np.uint32), want32.view(np.uint32))
    assert np.array_equal(run(dev, "f64", np.float64, k, elig).view(np.uint64), want.view(np.uint64))


def test_eligible_is_the_comparison(dev):
    # valid densities and fractions, both zeros, against every kind of threshold, NaNs of both signs among them
    dev.elig.argtypes = [C.c_double] * 3
    for n_th in (0.0, -0.0, 5e-324, 1e-6, 1.0, np.inf, np.nan, np.copysign(np.nan, -1.0)):
        for nh in (0.0, -0.0, 5e-324, 1e-6, np.nextafter(1e-6, 0), 1.0, 1e300):
            for x in (0.0, -0.0, 0.5, 1.0):
                assert bool(dev.elig(nh, x, n_th)) == (nh >= n_th and (1.0 - x) * nh > 0.0), (nh, x, n_th)
