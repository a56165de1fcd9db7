"""The reverse sweep of the RMHD dissipation through the closed-form waves against the one by
the Gram form's tangents (mhd_diss_vjp_gram), both built for the host, on random states with
distinct speeds; and the choice between them outside the closed form's range.

Bound: 1e-7 of the largest entry (gaps of 1e-3 and more: eps / 1e-3 for vectors, squared gaps in
the Gram tangents' quotients of quotients, times WENO weights of eps 1e-6)."""
import ctypes

import numpy as np
import pytest

import device_host
import oracle

SRC = r"""
#include "esmm_mhd_vjp.cuh"
using namespace esmm;
extern "C" int vjp(int form, double gam, double eps, const double *w, double Lk, double jt, const double *lrot,
                   const double (*TV)[8], double *out)
{
    Phys ph;
    ph.gamma = gam;
    ph.gm1i = 1.0 / (gam - 1.0);
    ph.igg = (gam - 1.0) / gam;
    ph.eps = eps;
    ph.sign_tol = 1e-10;
    double gTV[6][8], gw[8], Rz[8], hl;
    bool ok = true;
    if (form == 0) ok = mhd_diss_vjp_waves<5>(ph, w, Lk, jt, lrot, TV, gTV, gw, Rz, hl);
    else if (form == 1) mhd_diss_vjp_gram<5>(ph, w, Lk, jt, lrot, TV, gTV, gw, Rz, hl);
    else mhd_diss_vjp<5>(ph, w, Lk, jt, lrot, TV, gTV, gw, Rz, hl);
    if (!ok) return 0;
    for (int b = 0; b < 8; ++b) {
        for (int k = 0; k < 6; ++k) out[8 * k + b] = gTV[k][b];
        out[48 + b] = gw[b];
        out[56 + b] = Rz[b];
    }
    out[64] = hl;
    return 1;
}
"""
GAMMA = 5.0 / 3.0


@pytest.fixture(scope="module")
def dev(tmp_path_factory):
    return device_host.load(SRC, tmp_path_factory.mktemp("vjp"))


def _run(dev, form, w, lrot, TV, eps=1e-6):
    a = [np.ascontiguousarray(v, np.float64) for v in (w, lrot, TV)]
    out = np.zeros(65)
    p = [v.ctypes.data_as(ctypes.c_void_p) for v in a + [out]]
    ok = dev.vjp(form, ctypes.c_double(GAMMA), ctypes.c_double(eps), p[0], ctypes.c_double(1.1), ctypes.c_double(0.05), p[1],
                 p[2], p[3])
    return ok, out


def _state(r):
    return np.array([np.exp(r.uniform(-1, 1)), *r.uniform(-0.5, 0.5, 3), np.exp(r.uniform(-1, 1)), *r.uniform(-1.5, 1.5, 3)])


def _inputs(r, w):
    V = np.concatenate([oracle.mhd_entropy_vars(GAMMA, w * (1 + 0.1 * r.standard_normal(8))) for _ in range(6)]).reshape(6, 8)
    return r.standard_normal(8), V


def test_against_the_gram_form(dev):
    r = np.random.default_rng(1020)
    seen = 0
    while seen < 200:
        w = _state(r)
        if np.diff(oracle.mhd_eigen(GAMMA, w)[0][2:]).min() < 1e-3:
            continue
        seen += 1
        lrot, TV = _inputs(r, w)
        (a, x), (_, y), (_, z) = (_run(dev, f, w, lrot, TV) for f in (0, 1, 2))
        assert a == 1 and (x == z).all()
        for part in (slice(0, 48), slice(48, 56), slice(56, 64), slice(64, 65)):
            assert abs(x[part] - y[part]).max() <= 1e-7 * abs(y[part]).max(), (w, part)


@pytest.mark.parametrize("k", [-70, -50, 50, 70])
def test_outside_the_range(dev, k):
    r = np.random.default_rng(1021)
    s = np.array([4.0 ** k, 1, 1, 1, 4.0 ** k] + [2.0 ** k] * 3)     # rho, p and B
    t = np.array([1.0] * 5 + [2.0 ** k] * 3)                        # V
    for _ in range(50):
        w = _state(r)
        if np.diff(oracle.mhd_eigen(GAMMA, w)[0][2:]).min() < 1e-3:
            continue
        lrot, TV = _inputs(r, w)
        ref = _run(dev, 2, w, lrot, TV)[1]
        ok, _ = _run(dev, 0, w * s, lrot * t, TV * t, 1e-6 * 4.0 ** k)
        got = _run(dev, 2, w * s, lrot * t, TV * t, 1e-6 * 4.0 ** k)[1]
        assert ok == 0
        # -hl lrot.(R z) has the scale of lrot.U: 4^k with lrot t
        gT, gw = got[:48].reshape(6, 8) * t / 4.0 ** k, got[48:56] * s / 4.0 ** k
        assert abs(gT - ref[:48].reshape(6, 8)).max() <= 1e-7 * abs(ref[:48]).max()
        assert abs(gw - ref[48:56]).max() <= 1e-7 * abs(ref[48:56]).max()
