"""Two-dimensional bodies of many markers: up to 2432 a marker has a group of 16 lanes, above that of 4
(csrc/marker.cuh), at counts around that line and around full warps and blocks, on uniform and stretched
meshes, against the oracle (arXiv:1905.00182, Sec. 2, Eq. 7-11), with one marker off the grid.

Bounds, set before the first run, those of test_gpu_marker_groups.py.  Forces: |dF| <= 128 eps (|alpha xi|
+ beta (max|u| + |U|)).  Right-hand side: 64 eps of the split-flux scale and the spread-force scale per
element in FP64, 64 eps32 of the perturbation-flux scale and the spread-force scale RMS in the FP32 form.
"""
import dataclasses

import numpy as np
import pytest

from oracle import oracle as O
from paper_1905_00182_gb300 import workloads as W
from tests.test_gpu_stretched import case_2d

pytestmark = pytest.mark.gpu


def _case(nm, stretched):
    if stretched:
        c = case_2d(W.WENO5JS)
        spec = dataclasses.replace(c["spec"], max_markers=nm + 3)
        spec.src_amp = 0.0
        mesh, box, h = c["mesh"], 0.25, 0.04
    else:
        spec = W.GridSpec(dim=2, n=(61, 58, 1), lo=(-1.0,) * 3, hi=(1.0, 0.9, 1.0), gamma=1.4, Re=400.0,
                          qinf=W.freestream(2, 1.4), scheme=W.WENO5JS, max_markers=nm + 3)
        mesh, box, h = None, 0.8, spec.h[0]
    spec.alpha_pen, spec.beta_pen = W.penalty_defaults(h, 0.2 * h)
    Q = W.random_smooth_state(spec, seed=23, amp=2e-3)
    rnd = W.splitmix64(78 + nm, 4 * nm).reshape(4, nm)
    X = box * (2.0 * rnd[:2] - 1.0)
    U = 0.02 * (rnd[2:] - 0.5)
    dS = np.full(nm, 0.3 / nm)
    xi = 1e-3 * np.cos(np.arange(2 * nm)).reshape(2, nm)
    return spec, mesh, Q, X, U, dS, xi, h


@pytest.mark.parametrize("precision", [W.FP64, W.FP32_PERTURB])
@pytest.mark.parametrize("stretched", [False, True])
@pytest.mark.parametrize("nm,off", [(2432, None), (2433, None), (2464, 2463), (2501, 1207), (6000, 0)])
def test_many_markers_in_2d(nm, off, stretched, precision):
    from paper_1905_00182_gb300 import ibfsa as ib
    spec, mesh, Q, X, U, dS, xi, h = _case(nm, stretched)
    on = np.ones(nm, dtype=bool)
    if off is not None:
        X[1, off] = 40.0
        on[off] = False
    g = ib.Grid(dataclasses.replace(spec, precision=precision))
    for a in range(2):
        if mesh is not None:
            g.set_mesh(a, *mesh[a])
    g.set_state(Q)
    g.set_markers(X, U, dS)
    x = np.ascontiguousarray(xi)
    ib.ibfsa_set_penalty_integral(g.h, x.ctypes.data)
    L = g.rhs().cpu().numpy()
    F = g.marker_forces().cpu().numpy()
    assert g.status() == (0 if off is None else ib.IBFSA_STATUS_BOUNDS)
    g.rk3_step(0.2 * h, 1)
    xi1 = g.penalty_integral().cpu().numpy()
    g.close()
    Xo, Uo, So, xo = X[:, on], U[:, on], dS[on], xi[:, on]
    Lo, Fo = O.rhs(spec, Q, Xo, Uo, So, xo, return_markers=True, stretch=mesh)[:2]
    if off is not None:
        assert (F[:, off] == 0.0).all() and (xi1[:, off] == xi[:, off]).all()
    eps, eps32 = np.finfo(np.float64).eps, np.finfo(np.float32).eps
    umax = np.abs(Q[1:3] / Q[0]).max()
    assert np.all(np.abs(F[:, on] - Fo) <=
                  128 * eps * (np.abs(spec.alpha_pen * xo) + spec.beta_pen * (umax + np.abs(Uo))))
    fs = np.abs(Fo).max() * 0.25 * So.sum() / h ** 2
    alpha = O.wavespeeds(spec, Q)
    p = (spec.gamma - 1) * (Q[-1] - 0.5 * np.sum(Q[1:3] ** 2, axis=0) / Q[0])
    if precision == W.FP64:
        scale = (np.abs(Q[-1] + p).max() + max(alpha) * np.abs(Q).max()) / h
        assert np.abs(L - Lo).max() <= 64 * eps * (scale + fs)
    else:
        qinf = np.asarray(spec.qinf[:4]).reshape(-1, 1, 1, 1)
        scale = (1.0 + max(alpha)) * np.abs(Q - qinf).max() * 3.5 / h
        assert np.sqrt(np.mean((L - Lo) ** 2)) <= 64 * eps32 * (scale + fs)
