"""The RMHD scaled eigenvectors as the flux kernels form them (mhd_scaled_waves, built for
the host) against the oracle's Gram form, column by column up to sign: distinct speeds,
one and both sides with a pair of close speeds, pairs that the first two rows of the
canonical basis decide and pairs that they do not (v_1 B_1/sqrt(e) above 3/4), three and
four equal speeds, no field, fields down to the smallest numbers; FP64 and FP32.

Bound: the speeds of different clusters are at least 1e-2 apart here, so both sides'
vectors carry ~eps |C| / 1e-2 with a few operations' factor: 1e-11 in FP64, 2e-3 in FP32
(eps 6e-8, W up to 2.3)."""
import ctypes

import numpy as np
import pytest

import device_host
import oracle

SRC = r"""
#include "esmm_mhd.cuh"
using namespace esmm;
template <typename R> static void waves(double gam, const double *w, double *lohi, double *Rv)
{
    Phys ph;
    ph.gamma = gam;
    ph.gm1i = 1.0 / (gam - 1.0);
    ph.igg = (gam - 1.0) / gam;
    const double W = 1.0 / std::sqrt(1.0 - (w[1] * w[1] + w[2] * w[2] + w[3] * w[3]));
    R us[3], Bs[3], lo, hi, M[8][8];
    for (int k = 0; k < 3; ++k) {
        us[k] = (R)(W * w[1 + k]);
        Bs[k] = (R)w[5 + k];
    }
    mhd_scaled_waves<R>(ph, (R)w[0], (R)w[4], (R)(1.0 / w[4]), us, Bs, lo, hi, M);
    lohi[0] = lo;
    lohi[1] = hi;
    for (int m = 0; m < 8; ++m)
        for (int r = 0; r < 8; ++r) Rv[8 * m + r] = M[m][r];
}
extern "C" void waves64(double g, const double *w, double *l, double *R) { waves<double>(g, w, l, R); }
extern "C" void waves32(double g, const double *w, double *l, double *R) { waves<float>(g, w, l, R); }
"""
GAMMA = 5.0 / 3.0
BOUND = {"64": 1e-11, "32": 2e-3}


@pytest.fixture(scope="module")
def dev(tmp_path_factory):
    return device_host.load(SRC, tmp_path_factory.mktemp("waves"))


def production(dev, prec, w, gamma=GAMMA):
    w = np.ascontiguousarray(w, np.float64)
    lohi, R = np.zeros(2), np.zeros((8, 8))
    p = [a.ctypes.data_as(ctypes.c_void_p) for a in (w, lohi, R)]
    getattr(dev, "waves" + prec)(ctypes.c_double(gamma), *p)
    return lohi, R


def worst(R, ref):
    """largest difference of a column, up to its sign, relative to the column"""
    return np.max([np.minimum(abs(a - b).max(), abs(a + b).max()) / abs(b).max() for a, b in zip(R, ref)])   # (NaN: NaN)


def state(rho, v, p, B):
    return np.array([rho, *v, p, *B], float)


STATES = {
    "distinct": [state(1.0, (0.3, 0.2, -0.1), 0.8, (0.6, 0.5, 0.4)), state(0.4, (-0.5, 0.3, 0.6), 1.5, (-0.9, 0.7, 1.1))],
    "pairs": [state(1.0, (0.3, 0.0, 0.0), 0.1, (3.0, 1e-3 * np.cos(t), 1e-3 * np.sin(t))) for t in (0.0, 0.4, 0.8, 2.0)] +
             [state(1.0, (-0.2, 0.0, 0.1), 1.0, (0.7, 1e-3, 5e-4)), state(1.0, (0.2, 0.0, 0.0), 1.0, (-0.7, 0.0, 0.0))],
    "undecided pairs": [state(1.0, (v, 0.0, 0.0), 0.1, (b, 1e-3 * np.cos(t), 1e-3 * np.sin(t)))
                        for v, b in ((0.9, 3.0), (-0.9, 3.0), (0.9, -3.0)) for t in (0.4, 0.8, 1.2, 2.0, 4.0)],
    "four at v_n": [state(1.0, (0.3, 0.2, -0.1), 0.8, (0.0, 0.5, 0.4)), state(1.0, (0.3, 0.2, -0.1), 0.8, (1e-7, 0.5, -0.4))],
    "no field": [state(1.0, (0.3, 0.2, -0.1), 0.8, (0.0, 0.0, 0.0)), state(0.2, (0.0, 0.0, 0.0), 0.8, (0.0, 0.0, 0.0))],
}


@pytest.mark.parametrize("prec", ["64", "32"])
@pytest.mark.parametrize("kind", list(STATES))
def test_columns(dev, kind, prec):
    for w in STATES[kind]:
        lam, ref = oracle.mhd_eigen(GAMMA, w)
        lohi, R = production(dev, prec, w)
        eps = 1e-13 if prec == "64" else 1e-5
        assert abs(lohi - lam[[2, 7]]).max() <= eps, w
        assert worst(R, ref.T) <= BOUND[prec], (w, worst(R, ref.T))


@pytest.mark.parametrize("prec", ["64", "32"])
@pytest.mark.parametrize("along", [1.0, 1e-3, 0.0])
def test_columns_of_weak_fields(dev, prec, along):
    """Random gas, fields of any weakness in random directions, near the normal and on it
    (from 1e-8 on the slow and Alfven speeds of both sides are one cluster)."""
    r = np.random.default_rng(990)
    for e in range(8, 46 if prec == "32" else 320, 1 if prec == "32" else 4):
        for _ in range(8):
            d = r.standard_normal(3)
            d[1:] *= along
            w = state(np.exp(r.uniform(-1, 1)), r.uniform(-0.5, 0.5, 3), np.exp(r.uniform(-1, 1)), d * 10.0 ** -e)
            ref = oracle.mhd_eigen(GAMMA, w)[1]
            R = production(dev, prec, w)[1]
            assert worst(R, ref.T) <= BOUND[prec], (w, worst(R, ref.T))


@pytest.mark.parametrize("prec", ["64", "32"])
@pytest.mark.parametrize("wlo,whi,cold,b2", [(10, 20, (1e-4, 1e-3), (1, 30)), (10, 20, (1e-4, 1), (0.01, 10)), (1, 60, (1e-6, 1), (0.01, 100))])
def test_columns_of_fast_magnetized_gas(dev, prec, wlo, whi, cold, b2):
    """Norms of fast, cold, strongly magnetized states: positive, and in FP32 the columns'
    median error, W^2 eps ~ 1e-5 over the p/(rho h) that the sound speed resolves, below 5e-3 up to
    W = 20 (FP64 1e-6, which is the oracle's own at these)."""
    r = np.random.default_rng(991)
    err = []
    for _ in range(600):
        W, d, n = r.uniform(wlo, whi), r.standard_normal(3), r.standard_normal(3)
        v = d / np.linalg.norm(d) * np.sqrt(1.0 - 1.0 / W ** 2)
        rho = np.exp(r.uniform(-1, 1))
        p = rho * np.exp(r.uniform(*np.log(cold)))
        n /= np.linalg.norm(n)
        b = np.sqrt((rho + 2.5 * p) * np.exp(r.uniform(*np.log(b2))) / (1.0 / W ** 2 + (v @ n) ** 2))
        w = state(rho, v, p, b * n)
        lohi, R = production(dev, prec, w)
        assert np.isfinite(lohi).all() and np.isfinite(R).all(), w
        err.append(worst(R, oracle.mhd_eigen(GAMMA, w)[1].T))
    if whi <= 20:
        assert np.median(err) <= (5e-3 if prec == "32" else 1e-6)
