"""Primitive recovery of the GPU (an FP32 estimate, one FP64 step of third order, the
safeguarded loop elsewhere) over Lorentz factors 1 to 60, cold to hot gas and weak to
dominant fields: p of J U(prim) against prim.  Bound: f is evaluated to a few ulp of
E + p (RMHD: of E + Z, Z = rho h W^2), its slope is at least 1/5 at these Gamma, and the
rounding of E and m enters with factors below 4: 128 eps (E + p), 512 eps (E + Z).
States without a pressure are refused as before."""
import numpy as np
import pytest

from paper_2107_12027_gb300 import esmm
from paper_2107_12027_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
EPS = np.finfo(np.float64).eps


@pytest.mark.parametrize("phys", ["rhd", "rmhd"])
@pytest.mark.parametrize("gamma", [4.0 / 3.0, 5.0 / 3.0])
@pytest.mark.parametrize("wmax,cold", [(1.05, 1e-6), (3.0, 1e-2), (60.0, 1e-2)])
def test_round_trip(phys, gamma, wmax, cold):
    nx, ny = 64, 48
    r = wl.rng(970)
    sh = (ny, nx)
    W = 1.0 + (wmax - 1.0) * r.random(sh)
    d = r.standard_normal((3,) + sh)
    if phys == "rhd":
        d[2] = 0.0
    v = d / np.sqrt((d ** 2).sum(0)) * np.sqrt(1.0 - 1.0 / W ** 2)
    rho = np.exp(r.uniform(-7, 5, sh))
    p = rho * np.exp(r.uniform(np.log(cold), 5, sh))
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


@pytest.mark.parametrize("phys", ["rhd", "rmhd"])
def test_states_without_a_pressure_are_refused(phys):
    nx, ny = 8, 8
    x = wl.uniform_mesh(nx, ny)
    nv = 4 if phys == "rhd" else 8
    cons = np.zeros((nv, ny, nx))
    cons[0] = 1.0
    cons[1] = 0.3
    cons[3 if nv == 4 else 4] = 2.0
    cons[1, 3, 4] = 10.0         # |m| far above E: no admissible state
    J = np.ones((ny, nx))
    with esmm.Grid((nx, ny), phys=esmm.RHD if nv == 4 else esmm.RMHD) as g:
        with pytest.raises(Exception):
            g.rhs(cons, J, x)
