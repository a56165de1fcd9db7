"""Primitive recovery in any units (built for the host): rho, p, E, m times 2^2k and B times 2^k
scale the root exactly, so every result is that of the unscaled state to the bit, warm or cold
started; and the conversions over a power of two that the FP32 parts take, against the
product's own conversion."""
import ctypes

import numpy as np
import pytest

import device_host

SRC = r"""
#include "esmm_mhd.cuh"
using namespace esmm;
extern "C" int rhd(double g, const double *U, double p0, double *o)
{
    return cons2prim(g, U[0], U[1], U[2], U[3], p0, o[0], o[1], o[2], o[3], o[4]);
}
extern "C" int rmhd(double g, const double *U, double Z0, double *o) { return cons2prim_mhd(g, U, Z0, o, o[8]); }
extern "C" float narrow(double x, int k) { return d2f_scaled(x, k); }
extern "C" double widen(float x, int k) { return f2d_scaled(x, k); }
"""
SHIFTS = [-140, -60, -50, -26, -8, 8, 26, 30, 50, 60, 140]


@pytest.fixture(scope="module")
def dev(tmp_path_factory):
    lib = device_host.load(SRC, tmp_path_factory.mktemp("rec"))
    lib.narrow.restype, lib.widen.restype = ctypes.c_float, ctypes.c_double
    return lib


def _recover(f, gamma, U, start):
    U, o = np.ascontiguousarray(U, np.float64), np.zeros(9)
    st = f(ctypes.c_double(gamma), U.ctypes.data_as(ctypes.c_void_p), ctypes.c_double(start), o.ctypes.data_as(ctypes.c_void_p))
    return st, o


def _states(r, mhd, gamma, count):
    for _ in range(count):
        W, d = 1.0 + 59.0 * r.random() ** 4, r.standard_normal(3) * [1, 1, mhd]
        v = d / np.linalg.norm(d) * np.sqrt(1.0 - 1.0 / W ** 2)
        rho = np.exp(r.uniform(-5, 5))
        p = rho * np.exp(r.uniform(np.log(1e-5), 5))
        q = (rho + gamma / (gamma - 1.0) * p) * W ** 2
        if not mhd:
            yield np.array([rho * W, q * v[0], q * v[1], q - p]), p
            continue
        B = np.sqrt(p) * np.exp(r.uniform(-8, 1)) * r.standard_normal(3)
        B2, vB = B @ B, v @ B
        yield np.array([rho * W, *((q + B2) * v - vB * B), q - p + 0.5 * (B2 * (1.0 + v @ v) - vB ** 2), *B]), q


@pytest.mark.parametrize("phys", ["rhd", "rmhd"])
@pytest.mark.parametrize("k", SHIFTS)
def test_units(dev, phys, k):
    mhd, gamma = phys == "rmhd", 5.0 / 3.0
    if mhd and abs(k) > 60:
        k = int(np.sign(k)) * 100          # ((m.B)^2 ~ E^3 in FP64)
    sU = np.ldexp(1.0, [2 * k] * (5 if mhd else 4) + [k] * (3 if mhd else 0))
    sw = np.ldexp(1.0, [2 * k, 0, 0, 0, 2 * k, k, k, k, 2 * k] if mhd else [2 * k, 0, 0, 2 * k, 0, 0, 0, 0, 0])
    f = getattr(dev, phys)
    for U, root in _states(np.random.default_rng(995), mhd, gamma, 300):
        for start in (0.0, root * 1.01):
            a, x = _recover(f, gamma, U, start)
            b, y = _recover(f, gamma, U * sU, start * 4.0 ** k)
            assert a == b == 0
            assert (x * sw == y).all(), (U, k, x * sw - y)


def test_scaled_conversions(dev):
    r = np.random.default_rng(996)
    with np.errstate(over="ignore"):
        for k in (-890, -300, -127, -1, 0, 1, 24, 127, 300, 890):   # (x 2^k normal)
            for x in np.concatenate([r.standard_normal(50), [0.0, -0.0, 1.0, -2.0 ** 127, 2.0 ** -126, 2.0 - 2.0 ** -25, np.inf, -np.inf]]):
                y = np.ldexp(x, k)
                ref = np.float32(x)
                ref = ref if not 0.0 < abs(ref) < 2.0 ** -126 else ref * 0
                assert np.float32(dev.narrow(ctypes.c_double(y), k)).tobytes() == ref.tobytes()
                w = float(np.float32(x))
                assert np.float64(dev.widen(ctypes.c_float(w), k)).tobytes() == np.float64(np.ldexp(w, k)).tobytes()
            # outside FP32's range: 0 and infinity
            assert dev.narrow(ctypes.c_double(2.0 ** -60), 100) == 0.0
            assert dev.narrow(ctypes.c_double(-2.0 ** 60), -100) == -np.inf
            assert np.isnan(dev.narrow(ctypes.c_double(np.nan), k)) and np.isnan(dev.widen(ctypes.c_float(np.nan), k))
    assert dev.widen(ctypes.c_float(1.0), -1100) == 0.0 and dev.widen(ctypes.c_float(-1.0), 1100) == -np.inf
