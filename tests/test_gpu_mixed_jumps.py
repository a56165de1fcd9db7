"""A mixed-form right-hand side across jumps of the characteristic variables from 1e2 to 1e5 (cold
dense gas, random velocities) against the FP64 form: finite, and within 1e-4 of each component's
largest value at half the nodes (the two forms' switches take jumps of 1e-10 and 1e-5 of the terms that
form them as zero, so that single nodes may differ by their whole dissipation)."""
import numpy as np
import pytest

import oracle
from paper_2107_12027_gb300 import esmm
from paper_2107_12027_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("phys", [esmm.RHD, esmm.RMHD])
@pytest.mark.parametrize("w", [3, 5])
@pytest.mark.parametrize("rho", [1e2, 1e4, 1e5])
def test_large_jumps(phys, w, rho):
    nx, ny = 24, 20
    x, r = wl.uniform_mesh(nx, ny), wl.rng(1031)
    mhd = phys == esmm.RMHD
    prim = np.zeros((8 if mhd else 4, ny, nx))
    prim[0] = rho * (1.0 + 0.1 * r.random((ny, nx)))
    prim[1] = r.uniform(-0.6, 0.6, (ny, nx))
    prim[2] = r.uniform(-0.6, 0.6, (ny, nx))
    prim[4 if mhd else 3] = 1.0
    if mhd:
        prim[5:] = 0.3 * r.standard_normal((3, 1, 1))
    cfg = oracle.make_cfg(nx, ny, p=2, w=w, **({"phys": oracle.RMHD} if mhd else {}))
    cons, J = oracle.init_state(cfg, prim, x)
    out = []
    for prec in (esmm.FP64, esmm.MIXED):
        with esmm.Grid((nx, ny), p=2, w=w, phys=phys, precision=prec) as g:
            out.append(g.rhs(cons, J, x)[0])
    ref, got = out
    assert np.isfinite(got).all()
    for a in range(len(ref)):
        assert np.median(np.abs(got[a] - ref[a])) <= 1e-4 * max(np.abs(ref[a]).max(), 1e-30), a
