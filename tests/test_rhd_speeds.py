"""The acoustic speeds of the CFL pass (rhd_speeds, built for the host) up to the Lorentz factors
where rounding leaves v^2 = 1, against extended precision; and the square root by the short
reciprocal over sqrt's domain (2 ulp).  Bound: 1 - v^2 carries ~4 eps, its root 4 sqrt(eps)."""
import ctypes

import numpy as np
import pytest

import device_host

SRC = r"""
#include "esmm_device.cuh"
using namespace esmm;
extern "C" double root(double x) { return qsqrt(x); }
extern "C" void speeds(double v2, double c2, double vn, double *o)
{
    rhd_speeds(v2, c2, std::sqrt(c2), qrcp<double>(1.0 - v2 * c2), vn, o[0], o[1]);
}
"""


@pytest.fixture(scope="module")
def dev(tmp_path_factory):
    lib = device_host.load(SRC, tmp_path_factory.mktemp("speeds"))
    lib.root.restype = ctypes.c_double
    return lib


def test_root(dev):
    x = np.concatenate([10.0 ** np.random.default_rng(1050).uniform(-308, 308, 500), [1.0, 2.0 ** -1022, 2.0 ** 1023]])
    got = np.array([dev.root(ctypes.c_double(v)) for v in x])
    assert (abs(got - np.sqrt(x)) <= 2 * np.spacing(np.sqrt(x))).all()
    for v in (0.0, -0.0, 5e-324, 1e-310, np.inf):
        assert dev.root(ctypes.c_double(v)) == np.sqrt(v)
    assert np.isnan(dev.root(ctypes.c_double(-1.0))) and np.isnan(dev.root(ctypes.c_double(np.nan)))


@pytest.mark.parametrize("v2", [0.0, 0.5, 1.0 - 2.0 ** -40, 1.0 - 2.0 ** -52, 1.0 - 2.0 ** -53, 1.0])
@pytest.mark.parametrize("share", [0.0, 0.3, 1.0])
@pytest.mark.parametrize("c2", [1e-6, 0.2, 0.6])
def test_speeds(dev, v2, share, c2):
    vn, o = share * np.sqrt(v2), np.zeros(2)
    dev.speeds(ctypes.c_double(v2), ctypes.c_double(c2), ctypes.c_double(vn), o.ctypes.data_as(ctypes.c_void_p))
    L = np.longdouble
    V, C, N = L(v2), L(c2), L(vn)
    d = np.sqrt(max(L(0), (1 - V) * (1 - V * C - N * N * (1 - C))) * C)
    ref = [(N * (1 - C) - d) / (1 - V * C), (N * (1 - C) + d) / (1 - V * C)]
    assert np.isfinite(o).all() and abs(o - np.array(ref, float)).max() <= 4 * np.sqrt(np.finfo(float).eps)
