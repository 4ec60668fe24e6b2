"""Immersed-boundary kernels that give one group of lanes to each marker (csrc/marker.cuh), at
marker counts around the groups per warp and per block, and the z-chunks of the 3D viscous
march, against the oracle (arXiv:1905.00182, Sec. 2, Eq. 7-11).

Bounds, set before the first run.  Forces: F = alpha xi + beta (sum u w - U) in FP64 on both
sides from the same FP64 state; the 4^d weights sum to one and every product and addition is
rounded once, so |dF| <= 128 eps (|alpha xi| + beta (max|u| + |U|)).  Right-hand side: the bounds
of the forms (64 eps of the split-flux scale per element for the fast FP64 form; for the FP32
form 64 eps32 RMS of the perturbation-flux scale), with the spread force scale added.
"""
import dataclasses
import os
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

from oracle import oracle as O  # noqa: E402
from paper_1905_00182_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


def _case(dim, nm, n):
    lo, hi = (-1.0,) * 3, (1.0, 0.9, 1.1)
    spec = W.GridSpec(dim=dim, n=n, lo=lo, hi=hi, gamma=1.4, Re=400.0, qinf=W.freestream(dim, 1.4),
                      scheme=W.WENO5JS, max_markers=max(nm, 1) + 3)
    h = spec.h[0]
    spec.alpha_pen, spec.beta_pen = W.penalty_defaults(h, 0.2 * h)
    Q = W.random_smooth_state(spec, seed=21, amp=2e-3)
    rnd = W.splitmix64(77 + nm, 2 * dim * nm).reshape(2 * dim, nm)
    X = -0.55 + 1.1 * rnd[:dim]
    U = 0.02 * (rnd[dim:] - 0.5)
    dS = np.full(nm, 0.3 / nm)
    xi = 1e-3 * np.cos(np.arange(dim * nm)).reshape(dim, nm)
    return spec, Q, X, U, dS, xi


@pytest.mark.parametrize("precision", [W.FP64, W.FP32_PERTURB])
@pytest.mark.parametrize("dim,nm,n", [(2, 1, (23, 26, 1)), (2, 7, (24, 25, 1)), (2, 9, (40, 33, 1)),
                                      (2, 33, (31, 32, 1)), (3, 1, (12, 13, 11)),
                                      (3, 3, (14, 12, 13)), (3, 9, (33, 9, 17)),
                                      (3, 17, (20, 31, 70))])
def test_forces_and_spreading(dim, nm, n, precision):
    from paper_1905_00182_gb300 import ibfsa as ib
    spec, Q, X, U, dS, xi = _case(dim, nm, n)
    spec = dataclasses.replace(spec, precision=precision)
    Lo, Fo = O.rhs(spec, Q, X, U, dS, xi, return_markers=True)[:2]
    g = ib.Grid(spec)
    g.set_state(Q)
    g.set_markers(X, U, dS)
    x = np.ascontiguousarray(xi)
    ib.ibfsa_set_penalty_integral(g.h, x.ctypes.data)
    L = g.rhs().cpu().numpy()
    F = g.marker_forces().cpu().numpy()
    assert g.status() == 0
    g.close()
    eps = np.finfo(np.float64).eps
    umax = np.abs(Q[1:1 + dim] / Q[0]).max()
    bound = 128 * eps * (np.abs(spec.alpha_pen * xi) + spec.beta_pen * (umax + np.abs(U)))
    assert np.all(np.abs(F - Fo) <= bound)
    # scale of the spread force density (weights at most 1/2 per direction, all markers on a cell)
    fs = np.abs(Fo).max() * 0.5 ** dim * dS.sum() / np.prod(spec.h)
    alpha = O.wavespeeds(spec, Q)
    p = (spec.gamma - 1) * (Q[-1] - 0.5 * np.sum(Q[1:1 + dim] ** 2, axis=0) / Q[0])
    inv_h = 1.0 / min(spec.h)
    if precision == W.FP64:
        scale = (np.abs(Q[-1] + p).max() + max(alpha) * np.abs(Q).max()) * inv_h
        assert np.abs(L - Lo).max() <= 64 * eps * (scale + fs)
    else:
        qinf = np.asarray(spec.qinf[:dim + 2]).reshape(-1, 1, 1, 1)
        scale = (1.0 + max(alpha)) * np.abs(Q - qinf).max() * 3.5 * inv_h
        rms = np.sqrt(np.mean((L - Lo) ** 2))
        assert rms <= 64 * np.finfo(np.float32).eps * (scale + fs)
