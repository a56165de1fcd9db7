"""Mixed right-hand sides of fast (W = 10 to 20), cold (p/rho 1e-4 to 1e-3), strongly
magnetized gas (b^2 up to 30 rho h), rough in every variable: finite, and in the mean within
1e-2 of the oracle's (the FP32 eigenvectors are 6e-4 off in the median and 0.1 in the worst percent
of such states, and the dissipation is of the size of the whole).  WENO3: the fourth powers of
WENO5's weights leave FP32's range at differences of V this rough."""
import numpy as np
import pytest

import oracle
from paper_2107_12027_gb300 import esmm
from paper_2107_12027_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("direction", [(1.0, 0.2, 0.1), (-0.3, 1.0, 0.3), (0.5, 0.4, -0.8)])
def test_rhs(direction, p=1, w=3):
    nx, ny = 48, 40
    r = wl.rng(1001)
    sh = (ny, nx)
    W = r.uniform(10, 20, sh)
    d = np.array(direction)[:, None, None] + 0.02 * r.standard_normal((3,) + sh)
    v = d / np.sqrt((d ** 2).sum(0)) * np.sqrt(1.0 - 1.0 / W ** 2)
    rho = np.exp(r.uniform(-1, 1, sh))
    pr = rho * np.exp(r.uniform(np.log(1e-4), np.log(1e-3), sh))
    n = np.array([0.6, -0.5, 0.6])[:, None, None] + 0.1 * r.standard_normal((3,) + sh)
    b = np.sqrt((rho + 2.5 * pr) * np.exp(r.uniform(0, np.log(30), sh)) / ((n ** 2).sum(0) / W ** 2 + (v * n).sum(0) ** 2))
    prim = np.concatenate([np.stack([rho, v[0], v[1], v[2], pr]), b * n])
    x = wl.uniform_mesh(nx, ny)
    cfg = oracle.make_cfg(nx, ny, phys=oracle.RMHD, gamma=5.0 / 3.0, p=p, w=w)
    cons, J = oracle.init_state(cfg, np.ascontiguousarray(prim), x)
    ref = oracle.rhs(cfg, cons, J, x)[0]
    with esmm.Grid((nx, ny), gamma=5.0 / 3.0, p=p, w=w, phys=esmm.RMHD, precision=esmm.MIXED) as g:
        got = g.rhs(cons, J, x)[0]
    assert np.isfinite(got).all()
    for k in range(8):
        assert np.abs(got[k] - ref[k]).mean() <= 1e-2 * np.abs(ref[k]).mean(), k
