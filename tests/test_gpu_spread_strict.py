"""Strict IB interpolation and spreading (one table of supports, cells gathering their markers in
order) against the oracle, bit for bit (arXiv:1905.00182, Sec. 2, Eq. 7-11): marker counts around
a block of supports (8) and a ballot (256), clustered markers (many on one cell), markers spread
over several tiles, and a grid so small that its padded state holds the table of a few markers
only, so that the spreading runs in several passes."""
import os
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

from oracle import oracle as O  # noqa: E402
from paper_1905_00182_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n,nm,spread", [
    (2, (40, 37, 1), 1, 0.5), (2, (40, 37, 1), 9, 0.05), (2, (40, 37, 1), 257, 0.6),
    (2, (6, 7, 1), 200, 0.1), (3, (20, 19, 17), 8, 0.5), (3, (20, 19, 17), 300, 0.03),
    (3, (33, 18, 25), 513, 0.6), (3, (6, 6, 6), 900, 0.1)])
def test_bits(dim, n, nm, spread):
    from paper_1905_00182_gb300 import ibfsa as ib
    spec = W.GridSpec(dim=dim, n=n, lo=(-1.0,) * 3, hi=(1.0,) * 3, gamma=1.4, Re=300.0,
                      qinf=W.freestream(dim, 1.4), scheme=W.TENO5, max_markers=nm + 2)
    spec.alpha_pen, spec.beta_pen = W.penalty_defaults(spec.h[0], 0.2 * spec.h[0])
    Q = W.random_smooth_state(spec, seed=31, amp=2e-3)
    rnd = W.splitmix64(5 + nm, 2 * dim * nm).reshape(2 * dim, nm)
    X = spread * (2.0 * rnd[:dim] - 1.0)
    U = 0.02 * (rnd[dim:] - 0.5)
    dS = 0.3 / nm * (1.0 + np.arange(nm) / nm)
    xi = 1e-3 * np.cos(np.arange(dim * nm)).reshape(dim, nm)
    Lo, Fo = O.rhs(spec, Q, X, U, dS, xi, return_markers=True)[:2]
    g = ib.Grid(spec, strict=True)
    g.set_state(Q)
    g.set_markers(X, U, dS)
    x = np.ascontiguousarray(xi)
    ib.ibfsa_set_penalty_integral(g.h, x.ctypes.data)
    L = g.rhs().cpu().numpy()
    F = g.marker_forces().cpu().numpy()
    assert g.status() == 0
    g.close()
    assert np.array_equal(F, Fo)
    assert np.array_equal(L, Lo)
