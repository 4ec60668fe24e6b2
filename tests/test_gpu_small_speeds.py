"""Split speeds max |u_d| + c (the global Lax-Friedrichs splitting of arXiv:1905.00182, Sec. 2) where the
squared sound speed lies at and below FP32's smallest normal number, 1.2e-38: the fast FP64 form screens
the cells in FP32, and the maximum must be that of all cells.  One cell has the largest velocity and hardly
any sound speed, its neighbour the largest sum.  Bound, set before the first run: the speeds are a few
roundings of FP64 quantities, 16 eps.
"""
import numpy as np
import pytest

from paper_1905_00182_gb300 import workloads as W

pytestmark = pytest.mark.gpu

GAMMA = 1.4


@pytest.mark.parametrize("strict", [False, True])
@pytest.mark.parametrize("scale", [1e-24, 1e-21, 1e-20, 1e-19, 1e-18, 1e-13, 1e-12, 1e-11, 1.0, 1e18, 1e19, 1e25])
@pytest.mark.parametrize("dim", [2, 3])
def test_maximum_of_small_and_large_speeds(dim, scale, strict):
    from paper_1905_00182_gb300 import ibfsa as ib
    n = (15, 12, 1) if dim == 2 else (13, 9, 7)
    spec = W.GridSpec(dim=dim, n=n, lo=(0.0,) * 3, hi=(1.0,) * 3, gamma=GAMMA, Re=0.0,
                      qinf=W.freestream(dim, GAMMA), scheme=W.TENO5)
    r = W.splitmix64(3, (dim + 2) * int(np.prod(n))).reshape((dim + 2,) + tuple(reversed(n)))
    worst = 0.0
    for c_big in (0.3, 1.0):  # with scale 1e-19: c^2 = 9e-40 and 1e-38
        rho = 1.0 + 0.2 * r[0]
        u = 0.5 * scale * (r[1:1 + dim] - 0.5)
        c = 0.01 * scale * (1.0 + r[dim + 1])
        at = (0, 4, 5) if dim == 2 else (3, 4, 5)
        u[(slice(None),) + at] = scale             # the largest velocity
        beside = at[:2] + (at[2] + 1,)
        u[(slice(None),) + beside] = 0.9 * scale   # the largest sum
        c[beside] = c_big * scale
        p = rho * c * c / GAMMA
        Q = np.concatenate([rho[None], rho * u,
                            (p / (GAMMA - 1.0) + 0.5 * rho * np.sum(u * u, axis=0))[None]])
        g = ib.Grid(spec, strict=strict)
        g.set_state(Q)
        got = g.max_wavespeed()
        g.close()
        # the pressure comes back from the energy with the roundings of the kinetic energy
        back = (GAMMA - 1.0) * (Q[-1] - 0.5 * np.sum(Q[1:1 + dim] ** 2, axis=0) / Q[0])
        want = np.abs(Q[1:1 + dim] / Q[0]) + np.sqrt(np.maximum(GAMMA * back / Q[0], 0.0))
        for a in range(dim):
            worst = max(worst, abs(got[a] / want[a].max() - 1.0))
    assert worst <= 16 * np.finfo(np.float64).eps
