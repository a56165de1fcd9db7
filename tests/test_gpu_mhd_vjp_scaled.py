"""The RMHD vector-Jacobian product (2D, 3D) in units far from one: rho and p times 2^2k, B times
2^k and the WENO epsilon times 2^2k scale the right-hand side exactly, so the product with mu
over the components' scales is that of the unscaled state over them.  Beyond 1e25 and 1e-25 the
eigenvectors are the Gram form's and their tangents replace the reverse sweep.  Bound: 1e-8 of
each component's largest value (the Gram form's tangents, ~eps over the 1e-5 within which speeds
cluster, amplified by the WENO weights)."""
import numpy as np
import pytest

import oracle
from paper_2107_12027_gb300 import esmm
from paper_2107_12027_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
G43 = 4.0 / 3.0


def _product(n, k):
    d3 = len(n) == 3
    x = wl.wavy_mesh3(n, amp=0.03) if d3 else wl.wavy_mesh(*n, amp=0.03)
    r = wl.rng(1010)
    prim = wl.smooth_random_state_mhd3(x, r) if d3 else wl.smooth_random_state_mhd(x, r)
    cfg = oracle.make_cfg3(*n, gamma=G43, p=2, w=5) if d3 else oracle.make_cfg(*n, gamma=G43, p=2, w=5, phys=oracle.RMHD)
    cons, J = (oracle.init_state3 if d3 else oracle.init_state)(cfg, prim, x)
    s = np.array([4.0 ** k] * 5 + [2.0 ** k] * 3).reshape((8,) + (1,) * len(n))
    mu = r.standard_normal(cons.shape)
    with (esmm.Grid3(n, gamma=G43, p=2, w=5) if d3 else esmm.Grid(n, gamma=G43, p=2, w=5, phys=esmm.RMHD)) as g:
        g.set_params(weno_eps=1e-6 * 4.0 ** k)
        return g.rhs_vjp(np.ascontiguousarray(cons * s), J, x, None, mu / s) * s


@pytest.mark.parametrize("n", [(21, 16), (9, 8, 7)])
@pytest.mark.parametrize("k", [-70, -50, -30, 30, 50, 70])
def test_units(n, k):
    ref, got = _product(n, 0), _product(n, k)
    for a in range(8):
        assert np.abs(got[a] - ref[a]).max() <= 1e-8 * np.abs(ref[a]).max(), a
