"""The switch's decision in the FP64 form (built for the host).  Where FP32 decides (jump_sign), it
decides as FP64 does, over all of FP64's range and close to the threshold; and the whole dissipation
of one RHD and one RMHD interface is the same in any units: rho and p times 4^k, B times 2^k and
the WENO epsilon times 4^k scale it by 4^k (differences below 1e-20 of the epsilon need no scaled one: the
weights are the linear ones).  Bound: the jumps carry the rounding of the logarithms
(|ln 4^k| eps < 1e-13) through WENO weights of eps 1e-6: 1e-6 of the largest component."""
import ctypes

import numpy as np
import pytest

import device_host

SRC = r"""
#include "esmm_flux.cuh"
#include "esmm_mhd.cuh"
using namespace esmm;
static Phys phys(double gam, double eps)
{
    Phys ph;
    ph.gamma = gam;
    ph.gm1i = 1.0 / (gam - 1.0);
    ph.igg = (gam - 1.0) / gam;
    ph.eps = eps;
    ph.ln_thr = 1e-4;
    ph.sign_tol = 1e-10;
    return ph;
}
extern "C" int quick(double jump, double scale, float aT)   // (the term that aT belongs to: 0 at worst)
{
    float t[4] = {aT, 0.0f, 0.0f, 0.0f};
    jump_terms<double, 4>(t);
    return jump_sign(jump, 1e-10, d2f_int(scale) + t[3]);
}
extern "C" int full(double jump, double scale) { return jump_sign64(jump, 1e-10, scale); }
// six nodes (rho, v_x, v_y, p)
extern "C" void rhd(double gam, double eps, const double (*w)[4], double *F)
{
    const Phys ph = phys(gam, eps);
    double st[6][6];
    LmV<double> rho[6];
    for (int k = 0; k < 6; ++k) {
        const double W = 1.0 / std::sqrt(1.0 - w[k][1] * w[k][1] - w[k][2] * w[k][2]), beta = w[k][0] / w[k][3];
        const double s[6] = {beta, W * w[k][1], W * w[k][2], W, std::log(w[k][0]), std::log(beta)};
        for (int f = 0; f < 6; ++f) st[k][f] = s[f];
        rho[k].v = w[k][0];
        rho[k].l = s[4];
    }
    for (int a = 0; a < 4; ++a) F[a] = 0.0;
    const NodeStencil<double, ArrGet<double>> s{{st}};
    es_dissipation<double, 5>(0.8, 0.6, 0.05, rho[2], rho[3], s, ph, F);
}
// six nodes (rho, v, p, B), first axis along the normal
extern "C" void rmhd(double gam, double eps, const double (*w)[8], double *d)
{
    const Phys ph = phys(gam, eps);
    double V[6][8], us[3], Bs[3];
    for (int k = 0; k < 6; ++k) {
        const double W = 1.0 / std::sqrt(1.0 - w[k][1] * w[k][1] - w[k][2] * w[k][2] - w[k][3] * w[k][3]), beta = w[k][0] / w[k][4];
        double b0 = 0.0;
        for (int a = 0; a < 3; ++a) b0 += W * w[k][1 + a] * w[k][5 + a];
        V[k][0] = gam * ph.gm1i + std::log(w[k][0]) + ph.gm1i * std::log(beta) + beta;
        for (int a = 0; a < 3; ++a) {
            V[k][1 + a] = beta * W * w[k][1 + a];
            V[k][5 + a] = beta / W * (w[k][5 + a] + b0 * W * w[k][1 + a]);
        }
        V[k][4] = -beta * W;
    }
    const double (*l)[8] = w + 2, (*r)[8] = w + 3;
    for (int a = 0; a < 3; ++a) {
        us[a] = 0.6 * ((*l)[1 + a] + (*r)[1 + a]);
        Bs[a] = 0.5 * ((*l)[5 + a] + (*r)[5 + a]);
    }
    const double rho = 0.5 * ((*l)[0] + (*r)[0]), p = 0.5 * ((*l)[4] + (*r)[4]);
    es_dissipation_mhd<double, 5>(ph, rho, p, 1.0 / p, us, Bs, 1.1, 0.05, [=](int k, double v[8]) {
        for (int a = 0; a < 8; ++a) v[a] = V[k][a];
    }, d);
}
"""


@pytest.fixture(scope="module")
def dev(tmp_path_factory):
    return device_host.load(SRC, tmp_path_factory.mktemp("sign"))


def test_decision(dev):
    r = np.random.default_rng(1040)
    unsure = 0
    for e in range(-320, 300, 5):
        for _ in range(40):
            scale = 10.0 ** (e + 5 * r.random())
            f = r.choice([r.uniform(0.99, 1.01), 1.0 + r.uniform(-2e-3, 2e-3), 10.0 ** r.uniform(-20, 20), 0.0])
            jump = r.choice([-1.0, 1.0]) * scale * 1e-10 * f
            aT = 10.0 ** min(max(e + r.uniform(-3, 12), -44), 38)
            q = dev.quick(ctypes.c_double(jump), ctypes.c_double(scale), ctypes.c_float(aT))
            unsure += q == 2
            assert q == 2 or q == dev.full(ctypes.c_double(jump), ctypes.c_double(scale)), (jump, scale)
            if 1e-20 < scale < 1e10 and aT < 1e12 and not 0.998 < f < 1.002:
                assert q != 2
    assert unsure


@pytest.mark.parametrize("phys", ["rhd", "rmhd"])
@pytest.mark.parametrize("k", [-200, -166, -130, -70, -66, -50, 50, 66, 70])
def test_units(dev, phys, k):
    mhd = phys == "rmhd"
    nv = 8 if mhd else 4
    r = np.random.default_rng(1041)
    s = np.array([4.0 ** k] + [1.0] * (nv // 2 - 1) + [4.0 ** k] + [2.0 ** k] * 3) if mhd else np.array([4.0 ** k, 1, 1, 4.0 ** k])
    out_s = np.array([4.0 ** k] * 5 + [2.0 ** k] * 3)[:nv]

    def run(w, eps):
        w, F = np.ascontiguousarray(w), np.zeros(nv)
        getattr(dev, phys)(ctypes.c_double(5.0 / 3.0), ctypes.c_double(eps), w.ctypes.data_as(ctypes.c_void_p),
                           F.ctypes.data_as(ctypes.c_void_p))
        return F

    for _ in range(100):
        w = np.empty((6, nv))
        w[:, 0], w[:, nv // 2 if mhd else 3] = np.exp(r.uniform(-1, 1, (2, 6)))
        w[:, 1:nv // 2 if mhd else 3] = r.uniform(-0.4, 0.4, (6, 3 if mhd else 2))
        if mhd:
            w[:, 5:] = r.uniform(-1, 1, (6, 3))
        if k < -100:
            w[:] *= s ** (-80.0 / k)
            ref, got = run(w, 1e-6) / out_s ** (-80.0 / k), run(w * s ** (1.0 + 80.0 / k), 1e-6) / out_s
        else:
            ref, got = run(w, 1e-6), run(w * s, 1e-6 * 4.0 ** k) / out_s
        assert abs(got - ref).max() <= 1e-6 * abs(ref).max(), (ref, got)
