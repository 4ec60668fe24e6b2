"""The FP32 form's FP64 state: the update's conversions are done by integer operations.  A step from a
free stream with a pressure source gives increments from 1e-3 down through FP32's subnormal range to
zero (the Gaussian's tail), and the sponge reads the FP32 state back.  The FP64 state is the initial one
plus FP32 numbers: from q = 0 (the transverse momentum's free stream) it is an FP32 number to the bit, and
the rounded state taken over by the next step is the one that a grid rounds from the FP64 state itself
(set_state): two steps in one call and two calls with the state put back in between agree to the bit.
"""
import numpy as np
import pytest

from paper_1905_00182_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("re", [0.0, 100.0])
@pytest.mark.parametrize("n", [(67, 35), (40, 21, 19)])
def test_increments_of_every_size(n, re):
    from paper_1905_00182_gb300 import ibfsa as ib
    dim = len(n)
    spec = W.GridSpec(dim=dim, n=tuple(n) + (1,) * (3 - dim), lo=(-1.0,) * 3, hi=(1.0,) * 3,
                      gamma=1.4, Re=re, qinf=W.freestream(dim, 1.4), scheme=W.TENO5,
                      precision=W.FP32_PERTURB, sponge_cells=3, sponge_sigma=2.0)
    spec.src_amp, spec.src_b, spec.src_omega, spec.src_xc = 1e-2, 150.0, 4.0, (0.1, 0.0, 0.0)
    dt = 0.1 * min(spec.h)
    Q0 = np.broadcast_to(np.asarray(spec.qinf[:dim + 2]).reshape(-1, 1, 1, 1), spec.shape()).copy()

    def grid(Q, t):
        g = ib.Grid(spec)
        g.set_state(Q)
        g.set_time(t)
        return g

    g = grid(Q0, 0.0)
    g.rk3_step(dt, 1)
    one = g.get_state().cpu().numpy()
    g.rk3_step(dt, 1)
    two = g.get_state().cpu().numpy()
    g.close()
    v = one[2]
    assert np.array_equal(v, v.astype(np.float32).astype(np.float64)) and np.abs(v).max() > 1e-9
    tiny = np.abs(v[v != 0.0]).min()
    assert tiny < 1.1754944e-38, tiny
    g = grid(one, dt)
    g.rk3_step(dt, 1)
    assert np.array_equal(g.get_state().cpu().numpy(), two)
    assert g.status() == 0
    g.close()
