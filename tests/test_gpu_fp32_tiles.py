"""FP32 component-wise passes at the edges of their tiles -- x rows of up to 64 (or 32) cells, two
faces per lane, with the extra last face of a full row; y and z tiles of 15 cells, by tensor copies
where the x extent is a multiple of 4 and by plain loads otherwise -- against the oracle
(arXiv:1905.00182, Sec. 2).

On smooth modes of amplitude 2e-3 both sides evaluate the same reconstruction, so per element the
difference is rounding: a face flux of each direction takes a few dozen FP32 operations on values
up to the perturbation-flux scale s_a = (|F'| + alpha |q'|), and L is its difference over h:
|dL| <= 64 eps32 sum_a s_a / h_a, set before the first run.
"""
import os
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

from oracle import oracle as O  # noqa: E402
from paper_1905_00182_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu

SIZES = [(6, 5), (31, 16), (32, 17), (33, 15), (63, 31), (64, 14), (65, 30), (66, 9), (127, 8),
         (128, 33), (129, 46), (12, 64), (100, 35), (5, 6, 7), (32, 15, 16), (33, 17, 30),
         (64, 31, 14), (65, 14, 33), (96, 9, 10), (40, 16, 46)]


@pytest.mark.parametrize("scheme", [W.WENO5JS, W.TENO5])
@pytest.mark.parametrize("n", SIZES)
def test_tiles(n, scheme):
    from paper_1905_00182_gb300 import ibfsa as ib
    dim = len(n)
    spec = W.GridSpec(dim=dim, n=tuple(n) + (1,) * (3 - dim), lo=(-1.0,) * 3, hi=(1.0,) * 3,
                      gamma=1.4, Re=0.0, qinf=W.freestream(dim, 1.4, vel=(0.1, 0.05, -0.05)),
                      scheme=scheme, precision=W.FP32_PERTURB)
    Q = W.random_smooth_state(spec, seed=43, amp=2e-3, vel0=(0.1, 0.05, -0.05))
    Lo = O.rhs(spec, Q)
    Lo = Lo[0] if isinstance(Lo, tuple) else Lo
    alpha = O.wavespeeds(spec, Q)
    dq = np.abs(Q - np.asarray(spec.qinf[:dim + 2]).reshape(-1, 1, 1, 1)).max()
    g = ib.Grid(spec)
    g.set_state(Q)
    L = g.rhs().cpu().numpy()
    assert g.status() == 0
    g.close()
    # |F'| <= 3.5 |q'| (the Jacobian's largest entry, the enthalpy 1/(gamma - 1) + u^2/2 ~ 2.5, and
    # the pressure's part)
    bound = sum(64 * np.finfo(np.float32).eps * (3.5 + alpha[a]) * dq / spec.h[a]
                for a in range(dim))
    assert np.abs(L - Lo).max() <= bound
