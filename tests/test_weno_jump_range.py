"""The WENO jumps of the mixed form (weno5_jump, weno3_jump in FP32, built for the host) against
FP64 on the same differences, whose largest runs from 1e-6 to 1e6, with smooth and rough parts in one
stencil, for any WENO epsilon from 1e-10 up.  Bound: every e is a sum of squares of relative error
a few eps, the combinations are convex: 100 eps (6e-8) of the largest difference."""
import ctypes

import numpy as np
import pytest

import device_host

SRC = r"""
#include "esmm_device.cuh"
using namespace esmm;
extern "C" double jump(int w, int f32, const float *D, double eps)
{
    if (w == 5)
        return f32 ? weno5_jump<float>(D[0], D[1], D[2], D[3], D[4], (float)(4.0 * eps))
                   : weno5_jump<double>(D[0], D[1], D[2], D[3], D[4], 4.0 * eps);
    return f32 ? weno3_jump<float>(D[0], D[1], D[2], (float)eps) : weno3_jump<double>(D[0], D[1], D[2], eps);
}
"""


@pytest.fixture(scope="module")
def jump(tmp_path_factory):
    lib = device_host.load(SRC, tmp_path_factory.mktemp("jump"))
    lib.jump.restype = ctypes.c_double
    return lambda w, f32, D, eps: lib.jump(w, f32, D.ctypes.data_as(ctypes.c_void_p), ctypes.c_double(eps))


@pytest.mark.parametrize("w", [3, 5])
@pytest.mark.parametrize("eps", [1e-4, 1e-6, 1e-8, 1e-10])
def test_range(jump, w, eps):
    r = np.random.default_rng(1030)
    for big in 10.0 ** np.arange(-6, 6.1, 0.25):
        for _ in range(60):
            D = r.uniform(-1, 1, 5)
            D[r.random(5) < 0.4] *= 10.0 ** -r.uniform(2, 9)     # smooth parts
            D[r.random(5) < 0.2] = 0.0
            D = np.ascontiguousarray(D / max(abs(D).max(), 1e-30) * big, np.float32)
            ref = jump(w, 0, D, eps)
            assert abs(jump(w, 1, D, eps) - ref) <= 6e-6 * abs(D).max(), (D, ref)
