"""RMHD right-hand sides and their adjoint with fast cold flow along a strong field (v_1 =
0.9, B_1 = 3, p = 0.1, a tangential field of 1e-3): on both sides of the x_1 sweep the Alfven
and a magnetosonic speed cluster, and only one of the two pairs gets its canonical basis from
the first two rows (v_1 B_1/sqrt(e) > 3/4).  Against the oracle, whose basis comes from the whole
Gram matrix.  Bounds as in test_gpu_mhd_pairs.py (1e-8 of a component's largest value) and
test_gpu_mhd_adjoint_clusters.py (1e-5 of |mu| |d rhs|)."""
import numpy as np
import pytest

import oracle
from paper_2107_12027_gb300 import esmm
from paper_2107_12027_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
G = 5.0 / 3.0


def _primitives(shape, angle, r):
    s = [sum(r.uniform(-1, 1) * np.cos(2 * np.pi * (k * np.arange(shape[-1]) / shape[-1]) + r.uniform(0, 6))
             for k in (1, 2)) + 0.3 * r.standard_normal(shape) for _ in range(8)]
    one = np.ones(shape)
    return np.ascontiguousarray(np.stack([
        one + 0.02 * s[0], 0.9 + 0.002 * s[1], 2e-4 * s[2], 2e-4 * s[3], 0.1 + 0.002 * s[4], 3.0 + 0.01 * s[5],
        1e-3 * np.cos(angle) * (1 + 0.1 * s[6]), 1e-3 * np.sin(angle) * (1 + 0.1 * s[7])]))


@pytest.mark.parametrize("p,w", [(2, 5), (1, 3)])
@pytest.mark.parametrize("angle", [0.4, 0.8, 2.0])
def test_rhs(angle, p, w):
    nx, ny = 33, 10
    x = wl.uniform_mesh(nx, ny)
    cfg = oracle.make_cfg(nx, ny, phys=oracle.RMHD, gamma=G, p=p, w=w)
    cons, J = oracle.init_state(cfg, _primitives((ny, nx), angle, wl.rng(980)), x)
    ref = oracle.rhs(cfg, cons, J, x)[0]
    with esmm.Grid((nx, ny), gamma=G, p=p, w=w, phys=esmm.RMHD) as g:
        got = g.rhs(cons, J, x)[0]
    for k in range(8):
        assert np.abs(got[k] - ref[k]).max() <= 1e-8 * np.abs(ref[k]).max(), k


def test_rhs_3d():
    n = (17, 6, 5)
    x = wl.uniform_mesh3(n)
    cfg = oracle.make_cfg3(*n, gamma=G, p=2, w=5)
    cons, J = oracle.init_state3(cfg, _primitives(n[::-1], 0.8, wl.rng(981)), x)
    ref = oracle.rhs3(cfg, cons, J, x)[0]
    with esmm.Grid3(n, gamma=G, p=2, w=5) as g:
        got = g.rhs(cons, J, x)[0]
    for k in range(8):
        assert np.abs(got[k] - ref[k]).max() <= 1e-8 * np.abs(ref[k]).max(), k


@pytest.mark.parametrize("angle", [0.4, 0.8])
def test_vjp(angle):
    nx, ny = 17, 8
    x = wl.uniform_mesh(nx, ny)
    cfg = oracle.make_cfg(nx, ny, phys=oracle.RMHD, gamma=G, p=2, w=5)
    cons, J = oracle.init_state(cfg, _primitives((ny, nx), angle, wl.rng(982)), x)
    r = wl.rng(983)
    mu = r.standard_normal(cons.shape)
    d = r.standard_normal(cons.shape) * 1e-3 * np.abs(cons).reshape(8, -1).max(1)[:, None, None]
    h = 1e-4
    dr = (oracle.rhs(cfg, cons + h * d, J, x)[0] - oracle.rhs(cfg, cons - h * d, J, x)[0]) / (2 * h)
    with esmm.Grid((nx, ny), gamma=G, p=2, w=5, phys=esmm.RMHD) as g:
        lam = g.rhs_vjp(cons, J, x, None, mu)
    assert abs((lam * d).sum() - (mu * dr).sum()) <= 1e-5 * np.linalg.norm(mu) * np.linalg.norm(dr)
