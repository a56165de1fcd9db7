"""The RMHD vector-Jacobian product where wave speeds coincide at every interface:
gas without a field (the slow and Alfven speeds equal the entropy wave's) and a
field and velocity along x_1 on a uniform mesh (a degenerate pair in the x_1 sweep,
four equal speeds in the x_2 sweep).  Along directions that keep the degeneracy the
right-hand side is differentiable; lam . d is compared with central differences of
the oracle's right-hand side.  Bound: 1e-5 of |mu| |d rhs|, that of the other
direction checks (h = 1e-6 of the state leaves ~1e-8 of rounding and truncation; the
switch Y is frozen in lam, and a flip inside +-h changes the difference by a term
that vanishes with the jump it belongs to)."""
import numpy as np
import pytest

import oracle
from paper_2107_12027_gb300 import esmm
from paper_2107_12027_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("case,keep", [("hydro", (0, 1, 2, 3, 4)), ("aligned", (0, 1, 4, 5))])
def test_vjp_with_clustered_speeds(case, keep):
    nx, ny = 19, 14
    x = wl.wavy_mesh(nx, ny, amp=0.03) if case == "hydro" else wl.uniform_mesh(nx, ny)
    prim = wl.smooth_random_state_mhd(x, wl.rng(940))
    if case == "hydro":
        prim[5:] = 0.0
    else:
        prim[2:4] = 0.0
        prim[6:] = 0.0
    cfg = oracle.make_cfg(nx, ny, phys=oracle.RMHD, gamma=5.0 / 3.0, p=2, w=5)
    cons, J = oracle.init_state(cfg, prim, x)
    r = wl.rng(941)
    d = np.zeros_like(cons)
    for k in keep:
        d[k] = r.standard_normal(cons.shape[1:]) * np.abs(cons[k]).mean()
    mu = r.standard_normal(cons.shape)
    h = 1e-6
    dr = (oracle.rhs(cfg, cons + h * d, J, x)[0] - oracle.rhs(cfg, cons - h * d, J, x)[0]) / (2 * h)
    with esmm.Grid((nx, ny), gamma=5.0 / 3.0, p=2, w=5, phys=esmm.RMHD) as g:
        lam = g.rhs_vjp(cons, J, x, None, mu)
    assert np.isfinite(lam).all()
    assert abs((lam * d).sum() - (mu * dr).sum()) <= 1e-5 * np.linalg.norm(mu) * np.linalg.norm(dr)
