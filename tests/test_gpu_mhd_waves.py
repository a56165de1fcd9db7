"""RMHD right-hand sides where the closed-form waves change branch: fields along
the normal (b_t -> 0), normal fields that vanish, no field, coinciding sound and
Alfven speeds, weak fields and large Lorentz factors.

Bound: max(1e-12, 10 s) of each component's largest value, s the oracle's own
change under 1e-14 relative noise on its input (as in test_gpu_mhd.py); components
below 1e-8 of the largest one are held to that scale."""
import numpy as np
import pytest

import oracle
from paper_2107_12027_gb300 import esmm
from paper_2107_12027_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
G43 = 4.0 / 3.0


def _state(case, x, r):
    w = wl.smooth_random_state_mhd(x, r)
    w[1:4] *= 0.5
    if case == "along":            # B along x_1 up to 1e-9, gas nearly so
        w[6:8] *= 1e-9
        w[2:4] *= 1e-9
    elif case == "no_normal":      # B_1 = 0 in places of 1e-7, exactly 0 elsewhere
        w[5] = np.where(x[0] < 0.5, 0.0, 1e-7 * w[5])
    elif case == "hydro":
        w[5:] = 0.0
    elif case == "weak":
        w[5:] *= 1e-9
    elif case == "fast":           # W up to ~14
        w[1:4] *= 0.9975 / np.sqrt((w[1:4] ** 2).sum(0).max())
    elif case == "triple":         # c_s = c_A for a field along the normal, perturbed by 1e-4
        w[4] = 1.0 + 0.1 * (w[0] - w[0].mean())
        w[0] = 1.0
        w[1:4] = 0.0
        rh = w[0] + 4.0 * w[4]
        cs2 = G43 * w[4] / rh
        w[5] = np.sqrt(cs2 * rh / (1.0 - cs2))
        w[6:8] *= 1e-4
    return np.ascontiguousarray(w)


def _rel(a, b, scale):
    return max(np.abs(a[k] - b[k]).max() / scale[k] for k in range(len(scale)))


@pytest.mark.parametrize("case", ["along", "no_normal", "hydro", "weak", "fast", "triple"])
@pytest.mark.parametrize("pw", [(2, 5), (1, 3)])
def test_rhs_at_the_waves_branches(case, pw):
    nx, ny = 29, 23
    x = wl.wavy_mesh(nx, ny, amp=0.03)
    prim = _state(case, x, wl.rng(910))
    cfg = oracle.make_cfg(nx, ny, phys=oracle.RMHD, gamma=G43, p=pw[0], w=pw[1])
    cons, J = oracle.init_state(cfg, prim, x)
    ref = oracle.rhs(cfg, cons, J, x)[0]
    top = np.abs(ref).max()
    scale = np.maximum(np.abs(ref).reshape(8, -1).max(1), 1e-8 * top)
    s = 0.0
    for seed in (1, 2):
        r = wl.rng(920 + seed)
        other = oracle.rhs(cfg, cons * (1.0 + 1e-14 * r.standard_normal(cons.shape)), J, x)[0]
        s = max(s, _rel(other, ref, scale))
    with esmm.Grid((nx, ny), gamma=G43, p=pw[0], w=pw[1], phys=esmm.RMHD) as g:
        got = g.rhs(cons, J, x)[0]
        g.state_set_cons(cons, J, x)
        assert abs(g.cfl_dt() / oracle.cfl_dt(cfg, cons, J, x) - 1.0) <= 1e-12
    assert _rel(got, ref, scale) <= max(1e-12, 10.0 * s), (case, _rel(got, ref, scale), s)
