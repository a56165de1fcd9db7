"""RMHD with fields down to the smallest numbers: right-hand sides (FP64 and mixed) and FP64
vector-Jacobian products with a smooth random field scaled by 1e-10 to 1e-170, in random
directions and along x_1, against the oracle; and a mixed step of the example's vortex, whose
field falls off as exp(-r^2/2) and passes through every size towards the corners.

Bounds: FP64 max(1e-12, 10 s) of each component's largest value as in
test_gpu_mhd_waves.py (s the oracle's change under 1e-14 relative noise, components below 1e-8
of the largest one held to that scale); mixed 5e-3 of each component, that of the mixed
right-hand sides (test_gpu_mhd_mixed.py), the field's components against the gas's; the
product's gas components 1e-7 (rounding over the cluster tolerance, 1e-11, through WENO weights that
amplify it up to ~1e3 times); the vortex's primitives after one step within 1e-4 of the FP64 step's,
about 1e-2 of what the step changes."""
import numpy as np
import pytest

import oracle
from paper_2107_12027_gb300 import esmm
from paper_2107_12027_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
G43 = 4.0 / 3.0
NX, NY = 29, 23


def _setup(scale, along):
    x = wl.wavy_mesh(NX, NY, amp=0.0 if along else 0.03)
    prim = wl.smooth_random_state_mhd(x, wl.rng(995))
    prim[1:4] *= 0.5
    if along:
        prim[6:8] = 0.0
    prim[5:8] *= scale
    cfg = oracle.make_cfg(NX, NY, phys=oracle.RMHD, gamma=G43, p=2, w=5)
    cons, J = oracle.init_state(cfg, np.ascontiguousarray(prim), x)
    return x, cfg, cons, J


SCALES = [1e-10, 1e-14, 1e-16, 1e-18, 1e-19, 1e-20, 1e-21, 1e-22, 1e-30, 1e-41, 1e-150, 1e-155, 1e-158, 1e-160, 1e-170]


@pytest.mark.parametrize("along", [False, True])
@pytest.mark.parametrize("scale", SCALES)
def test_rhs(scale, along):
    x, cfg, cons, J = _setup(scale, along)
    ref = oracle.rhs(cfg, cons, J, x)[0]
    size = np.maximum(np.abs(ref).reshape(8, -1).max(1), 1e-8 * np.abs(ref).max())
    s = 0.0
    for seed in (1, 2):
        r = wl.rng(996 + seed)
        other = oracle.rhs(cfg, cons * (1.0 + 1e-14 * r.standard_normal(cons.shape)), J, x)[0]
        s = max(s, (np.abs(other - ref).reshape(8, -1).max(1) / size).max())
    for prec, bound in ((esmm.FP64, max(1e-12, 10 * s)), (esmm.MIXED, 5e-3)):
        with esmm.Grid((NX, NY), gamma=G43, p=2, w=5, phys=esmm.RMHD, precision=prec) as g:
            got = g.rhs(cons, J, x)[0]
        for k in range(8):
            unit = size[k] if prec == esmm.FP64 or k < 5 else np.abs(ref).max()
            assert np.abs(got[k] - ref[k]).max() <= bound * unit, (k, prec)


@pytest.mark.parametrize("scale", [1e-19, 1e-155, 1e-158, 1e-160])
def test_vjp(scale):
    """... tends to the product without a field (checked in test_gpu_mhd_adjoint_clusters.py)."""
    mu = wl.rng(999).standard_normal((8, NY, NX))
    lam = []
    for sc in (scale, 0.0):
        x, cfg, cons, J = _setup(sc, False)
        with esmm.Grid((NX, NY), gamma=G43, p=2, w=5, phys=esmm.RMHD) as g:
            lam.append(g.rhs_vjp(cons, J, x, None, mu))
    assert np.isfinite(lam[0]).all()
    assert np.abs(lam[0][:5] - lam[1][:5]).max() <= 1e-7 * np.abs(lam[1][:5]).max()


@pytest.mark.parametrize("n", [40, 160])
def test_mixed_vortex_step(n):
    x = wl.uniform_mesh(n, n, (-5, -5), (5, 5))
    prim = wl.rmhd_vortex(x)
    out = {}
    for prec in (esmm.FP64, esmm.MIXED):
        with esmm.Grid((n, n), (-5, -5), (5, 5), gamma=5.0 / 3.0, p=2, w=5, phys=esmm.RMHD, precision=prec) as g:
            g.state_set(prim, x)
            if prec == esmm.FP64:
                dt = g.rk_step()
            else:
                g.rk_step(dt)
            out[prec] = g.state_get(esmm.GET_PRIM)
    assert np.isfinite(out[esmm.MIXED]).all()
    assert np.abs(out[esmm.MIXED] - out[esmm.FP64]).max() <= 1e-4
