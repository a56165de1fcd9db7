"""Right-hand sides in units far from one: rho and p times 4^k, B times 2^k and the WENO epsilon times
4^k scale them by 4^k (the induction's by 2^k), whatever power a short reciprocal's argument then has.
Bound: the logarithms' rounding, |ln 4^k| eps < 2e-14, through WENO weights of eps 1e-6: 1e-6 of each component's largest
value in FP64; the mixed form (2e-6 in the logarithms) within 1e-3 at half the nodes."""
import numpy as np
import pytest

import oracle
from paper_2107_12027_gb300 import esmm
from paper_2107_12027_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _state(kind):
    r = wl.rng(1060)
    if kind == "rmhd3":
        x = wl.wavy_mesh3((9, 8, 7), amp=0.03)
        cfg, prim = oracle.make_cfg3(9, 8, 7, p=2, w=5), wl.smooth_random_state_mhd3(x, r)
        return x, *oracle.init_state3(cfg, prim, x)
    x = wl.wavy_mesh(21, 16, amp=0.03)
    mhd = kind == "rmhd"
    cfg = oracle.make_cfg(21, 16, p=2, w=5, **({"phys": oracle.RMHD} if mhd else {}))
    return x, *oracle.init_state(cfg, (wl.smooth_random_state_mhd if mhd else wl.smooth_random_state)(x, r), x)


def _rhs(kind, k, prec):
    x, cons, J = _state(kind)
    s = np.array([4.0 ** k] * (4 if kind == "rhd" else 5) + [2.0 ** k] * (0 if kind == "rhd" else 3)).reshape((-1,) + (1,) * J.ndim)
    if kind == "rmhd3":
        grid = esmm.Grid3((9, 8, 7), p=2, w=5)
    else:
        grid = esmm.Grid((21, 16), p=2, w=5, phys=esmm.RMHD if kind == "rmhd" else esmm.RHD, precision=prec)
    with grid as g:
        g.set_params(weno_eps=1e-6 * 4.0 ** k)
        return g.rhs(np.ascontiguousarray(cons * s), J, x)[0] / s


@pytest.mark.parametrize("kind", ["rhd", "rmhd", "rmhd3"])
@pytest.mark.parametrize("k", [-66, -50, -30, 30, 50, 66])
def test_fp64(kind, k):
    ref, got = _rhs(kind, 0, esmm.FP64), _rhs(kind, k, esmm.FP64)
    for a in range(len(ref)):
        assert np.abs(got[a] - ref[a]).max() <= 1e-6 * np.abs(ref[a]).max(), a


@pytest.mark.parametrize("kind", ["rhd", "rmhd"])
@pytest.mark.parametrize("k", [-8, 8, 14])
def test_mixed(kind, k):
    ref, got = _rhs(kind, 0, esmm.FP64), _rhs(kind, k, esmm.MIXED)
    assert np.isfinite(got).all()
    for a in range(len(ref)):
        assert np.median(np.abs(got[a] - ref[a])) <= 1e-3 * np.abs(ref[a]).max(), a
