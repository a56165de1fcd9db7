"""The RMHD right-hand side where the Alfven and a magnetosonic speed of one side
cluster at every interface (a field along x_1 with a tangential part of 1e-3 and
less: gaps below 1e-6, well under the clustering threshold 1e-5, in the x_1 sweep; in
the x_2 sweep the slow and Alfven waves of both sides meet at v_2), against the
oracle, which builds the basis from the whole Gram matrix.  Bound: 1e-8 of the largest
component in FP64 (the Gram form's columns are good to ~1e-9 in its worst cases);
5e-3 in the mixed form, the bound of the mixed right-hand sides elsewhere (the switch Y
may differ at jumps of FP32 rounding size)."""
import numpy as np
import pytest

import oracle
from paper_2107_12027_gb300 import esmm
from paper_2107_12027_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("p,w", [(2, 5), (1, 3)])
@pytest.mark.parametrize("tangential,v3", [(0.0, 0.0), (1e-3, 0.0), (1e-3, 0.3), (1e-6, -0.3)])
def test_rhs_with_paired_speeds(p, w, tangential, v3, prec):
    nx, ny = 33, 18
    x = wl.uniform_mesh(nx, ny)
    prim = wl.smooth_random_state_mhd(x, wl.rng(960))
    s = wl.rng(961).standard_normal((2,) + prim.shape[1:])
    prim[2] = 0.1 * tangential * s[0]
    prim[3] = v3
    prim[5] = 0.7
    prim[6] = tangential * s[1]
    prim[7] = tangential * s[0]
    cfg = oracle.make_cfg(nx, ny, phys=oracle.RMHD, gamma=5.0 / 3.0, p=p, w=w)
    cons, J = oracle.init_state(cfg, prim, x)
    ref = oracle.rhs(cfg, cons, J, x)[0]
    with esmm.Grid((nx, ny), gamma=5.0 / 3.0, p=p, w=w, phys=esmm.RMHD,
                   precision=esmm.MIXED if prec == "mixed" else esmm.FP64) as g:
        got = g.rhs(cons, J, x)[0]
    assert np.abs(got - ref).max() <= (5e-3 if prec == "mixed" else 1e-8) * np.abs(ref).max()
