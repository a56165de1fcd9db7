"""The reciprocal and reciprocal square root of the flux kernels against IEEE division
and square root in FP64, over 60 binades and at their edges.  Bounds: 2 ulp = 2^-51 in
FP64 (first approximation below 2^-20, cubed below 2^-57, then the roundings of the
residual, of the correction and of the result: under 1.5 ulp); in FP32 the reciprocal
of a first approximation good to 2^-22 squared, 1.5 ulp, bounded by 2^-22."""
import ctypes
import pathlib
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SRC = r"""
#include "esmm_device.cuh"
using namespace esmm;
__global__ void k(const double *x, double *r, double *y, float *f, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    r[i] = qrcp<double>(x[i]);
    y[i] = qrsq<double>(x[i] < 0.0 ? -x[i] : x[i]);
    f[i] = qrcp<float>((float)x[i]);
}
extern "C" int run(const double *x, double *r, double *y, float *f, int n)
{
    double *dx, *dr, *dy;
    float *df;
    cudaMalloc(&dx, n * 8); cudaMalloc(&dr, n * 8); cudaMalloc(&dy, n * 8); cudaMalloc(&df, n * 4);
    cudaMemcpy(dx, x, n * 8, cudaMemcpyHostToDevice);
    k<<<(n + 127) / 128, 128>>>(dx, dr, dy, df, n);
    cudaMemcpy(r, dr, n * 8, cudaMemcpyDeviceToHost);
    cudaMemcpy(y, dy, n * 8, cudaMemcpyDeviceToHost);
    cudaMemcpy(f, df, n * 4, cudaMemcpyDeviceToHost);
    cudaFree(dx); cudaFree(dr); cudaFree(dy); cudaFree(df);
    return (int)cudaGetLastError();
}
"""


def test_reciprocals(tmp_path):
    csrc = pathlib.Path(__file__).resolve().parents[1] / "paper_2107_12027_gb300" / "csrc"
    (tmp_path / "k.cu").write_text(SRC)
    so = tmp_path / "k.so"
    subprocess.run(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-shared", "-Xcompiler",
                    "-fPIC", "-I", str(csrc), "-I", str(csrc.parents[1] / "include"), "-o", str(so),
                    str(tmp_path / "k.cu")], check=True)
    lib = ctypes.CDLL(str(so))
    r = np.random.default_rng(950)
    x = (1.0 + r.random(200000)) * 2.0 ** r.integers(-30, 30, 200000)
    edge = 2.0 ** np.arange(-60.0, 60.0)
    x = np.concatenate([x * r.choice([-1.0, 1.0], x.size), edge, np.nextafter(edge, 0.0), np.nextafter(edge, np.inf)])
    o, y, f = np.empty_like(x), np.empty_like(x), np.empty(x.size, np.float32)
    p = [a.ctypes.data_as(ctypes.c_void_p) for a in (x, o, y, f)]
    assert lib.run(*p, ctypes.c_int(x.size)) == 0
    assert abs(o * x - 1.0).max() <= 2.0 ** -51
    assert abs(y * np.sqrt(abs(x)) - 1.0).max() <= 2.0 ** -51
    x32 = x.astype(np.float32).astype(np.float64)
    assert abs(f * x32 - 1.0).max() <= 2.0 ** -22
