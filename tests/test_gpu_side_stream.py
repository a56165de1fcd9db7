"""The second sweep direction on its own stream: right-hand sides and steps equal those
with the directions in line (which timing the flux launches asks for) to the last
bit, repeatedly, and repeat themselves on a caller's stream."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2107_12027_gb300 import esmm  # noqa: E402
from paper_2107_12027_gb300 import workloads as wl  # noqa: E402

pytestmark = pytest.mark.gpu
MASK = (1 << esmm.KIND_IFACE) | (1 << esmm.KIND_PAIRS)


def _grid(kind, **kw):
    if kind == "rmhd3":
        n = (12, 10, 9)
        x = wl.wavy_mesh3(n, amp=0.03)
        return esmm.Grid3(n, **kw), wl.smooth_random_state_mhd3(x, wl.rng(980)), x
    x = wl.wavy_mesh(37, 26, amp=0.03)
    if kind == "rmhd":
        return esmm.Grid((37, 26), phys=esmm.RMHD, **kw), wl.smooth_random_state_mhd(x, wl.rng(981)), x
    return (esmm.Grid((37, 26), sweep=esmm.SWEEP_SPLIT if kind == "split" else esmm.SWEEP_FUSED, **kw),
            wl.smooth_random_state(x, wl.rng(982)), x)


@pytest.mark.parametrize("kind", ["fused", "split", "rmhd", "rmhd3"])
def test_equal_to_directions_in_line(kind):
    out = []
    for timed in (False, True):
        g, prim, x = _grid(kind)
        with g:
            g.state_set(prim, x)
            if timed:
                g.profile(MASK)
            cons, J = g.state_get(esmm.GET_CONS), g.state_get(esmm.GET_J)
            r = [g.rhs(cons, J, x)[0] for _ in range(5)]
            dts = [g.rk_step() for _ in range(3)]
            out.append((r, dts, g.state_get(esmm.GET_CONS)))
    for a in out[0][0] + out[1][0]:
        assert np.array_equal(a, out[0][0][0])
    assert out[0][1] == out[1][1]
    assert np.array_equal(out[0][2], out[1][2])


def test_on_a_callers_stream():
    s = torch.cuda.Stream()
    g, prim, x = _grid("fused", stream=s.cuda_stream)
    with g:
        g.state_set(prim, x)
        dev = dict(device="cuda", dtype=torch.float64)
        cons = torch.tensor(g.state_get(esmm.GET_CONS), **dev)
        J, xt = torch.tensor(g.state_get(esmm.GET_J), **dev), torch.tensor(x, **dev)
        oc, oj = torch.empty_like(cons), torch.empty_like(J)
        torch.cuda.synchronize()
        g.rhs(cons, J, xt, None, oc, oj)
        s.synchronize()
        ref = oc.clone()
        for _ in range(10):
            oc.zero_()
            torch.cuda.synchronize()
            g.rhs(cons, J, xt, None, oc, oj)
            s.synchronize()
            assert torch.equal(oc, ref)
