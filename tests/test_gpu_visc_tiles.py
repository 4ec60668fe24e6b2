"""Viscous terms of the 2D forms at the edges of the FP32 kernel's 64 x 16 tiles (its flux box reaches
two cells beyond), and of the FP64 fast form whose divergence is taken by the update kernel, on
uniform and stretched meshes, against the oracle (arXiv:1905.00182, Sec. 2).

Bound per element, set before the first run.  The state is smooth, of amplitude 2e-3, so both sides
evaluate the same formulas and differ by rounding.  Convective part: 64 eps sum_a s_a / h_a with
s_a = (3.5 + alpha_a) |q'| in FP32 (the perturbation form's rounding scale) and the whole flux,
3.5 + alpha_a, in FP64.  Viscous part: two nested fourth-order differences, each at most 1.5 |.| / h,
of velocities |u'| <= |q'| / rho (for FP64 the differences cancel the mean, its rounding stays: |u|);
a momentum component sums at most 4 such terms per pair of directions with weights up to 4/3, the
energy the same times |u|: 64 eps (16/3) (1/Re) sum_ab (1.5/h_a)(1.5/h_b) |u'|.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1905_00182_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SIZES = [(6, 5), (33, 15), (60, 16), (63, 17), (64, 16), (64, 33), (65, 18), (66, 31), (127, 12),
         (128, 32), (129, 34), (200, 7)]


@pytest.mark.parametrize("precision", [W.FP32_PERTURB, W.FP64])
@pytest.mark.parametrize("stretched", [False, True])
@pytest.mark.parametrize("n", SIZES)
def test_viscous_tiles(n, stretched, precision):
    from paper_1905_00182_gb300 import ibfsa as ib
    vel = (0.1, 0.05)
    spec = W.GridSpec(dim=2, n=tuple(n) + (1,), lo=(-1.0,) * 3, hi=(1.0,) * 3, gamma=1.4, Re=40.0,
                      qinf=W.freestream(2, 1.4, vel=vel), scheme=W.TENO5, precision=precision)
    Q = W.random_smooth_state(spec, seed=47, amp=2e-3, vel0=vel)
    h, mesh = list(spec.h), None
    if stretched:  # x = xi + 0.3 sin(pi xi) / pi in both directions: dx/dxi between 0.7 and 1.3 h
        mesh = []
        for a in range(2):
            xi = -1.0 + (np.arange(-4, n[a] + 4) + 0.5) * h[a]
            mesh.append((xi + 0.3 * np.sin(np.pi * xi) / np.pi,
                         h[a] * (1.0 + 0.3 * np.cos(np.pi * xi))))
            h[a] = mesh[a][1].min()
    Lo = O.rhs(spec, Q, stretch=mesh)
    Lo = Lo[0] if isinstance(Lo, tuple) else Lo
    g = ib.Grid(spec)
    for a in range(2):
        if mesh:
            g.set_mesh(a, *mesh[a])
    g.set_state(Q)
    L = g.rhs().cpu().numpy()
    assert g.status() == 0
    g.close()
    fp32 = precision == W.FP32_PERTURB
    eps = np.finfo(np.float32 if fp32 else np.float64).eps
    alpha = O.wavespeeds(spec, Q)
    dq = np.abs(Q - np.asarray(spec.qinf[:4]).reshape(-1, 1, 1, 1)).max()
    scale, du = (dq, dq / 0.9) if fp32 else (1.0, 0.2)
    bound = 64 * eps * sum((3.5 + alpha[a]) * scale / h[a] for a in range(2))
    bound += 64 * eps * 16 / 3 / spec.Re * du * sum(2.25 / (h[a] * h[b]) for a in range(2)
                                                    for b in range(2))
    assert np.abs(L - Lo).max() <= bound
