"""Primitive recovery of the GPU in units far from one: the states and the bound of
test_gpu_recovery.py (128 eps of E + p, RMHD 512 eps of E + Z), rho and p times 4^k (1e-30 to
1e30), B times 2^k."""
import numpy as np
import pytest

from paper_2107_12027_gb300 import esmm
from paper_2107_12027_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
EPS = np.finfo(np.float64).eps


@pytest.mark.parametrize("phys", ["rhd", "rmhd"])
@pytest.mark.parametrize("k", [-50, -33, -17, 17, 33, 50])
def test_round_trip(phys, k):
    nx, ny, gamma = 64, 48, 5.0 / 3.0
    r = wl.rng(971)
    sh = (ny, nx)
    W = 1.0 + 2.0 * r.random(sh)
    d = r.standard_normal((3,) + sh)
    if phys == "rhd":
        d[2] = 0.0
    v = d / np.sqrt((d ** 2).sum(0)) * np.sqrt(1.0 - 1.0 / W ** 2)
    rho = np.exp(r.uniform(-7, 5, sh)) * 4.0 ** k
    p = rho * np.exp(r.uniform(np.log(1e-2), 5, sh))
    rhoh = rho + gamma / (gamma - 1.0) * p
    if phys == "rhd":
        prim, kind = np.stack([rho, v[0], v[1], p]), esmm.RHD
        scale = 128 * (rhoh * W ** 2 + p)
    else:
        B = np.sqrt(p) * np.exp(r.uniform(-8, 1, sh)) * r.standard_normal((3,) + sh)
        prim, kind = np.concatenate([np.stack([rho, v[0], v[1], v[2], p]), B]), esmm.RMHD
        scale = 512 * (2 * rhoh * W ** 2 + (B ** 2).sum(0))
    with esmm.Grid((nx, ny), gamma=gamma, phys=kind) as g:
        g.state_set(np.ascontiguousarray(prim), wl.uniform_mesh(nx, ny))
        got = g.state_get(esmm.GET_PRIM)
    i = 3 if phys == "rhd" else 4
    assert np.isfinite(got).all()
    assert (abs(got[i] - p) / scale).max() <= EPS
