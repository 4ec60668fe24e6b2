"""The FP64 x pass takes 32 lines to a tile, the rows of a plane or, where these leave many lanes idle,
segments of rows of all planes: grids of few rows, rows that wrap over planes and segments, a short last
segment in any place of a tile, with 1, 2 and 4 faces per thread, against the oracle (arXiv:1905.00182, Sec. 2), with the states and bounds of test_gpu_conv_tiles.py.
"""
import dataclasses

import numpy as np
import pytest

from oracle import oracle as O
from paper_1905_00182_gb300 import workloads as W
from tests.test_gpu_conv_tiles import _rhs, _spec, _state

pytestmark = pytest.mark.gpu

SIZES = [(2000, 1), (2000, 8), (4000, 33), (64, 9, 100), (301, 2), (1000, 3), (67, 5), (513, 8), (33, 17),
         (95, 31), (64, 96), (29, 45), (200, 1, 1), (120, 3, 5), (61, 9, 7), (34, 5, 13), (8, 33, 3),
         (97, 2, 31)]


@pytest.mark.parametrize("scheme", [W.WENO5JS, W.TENO5])
@pytest.mark.parametrize("walls", [W.BC_ZERO_GRAD, W.BC_CHARACTERISTIC])
@pytest.mark.parametrize("n", SIZES)
def test_strict_bits(n, walls, scheme):
    spec = dataclasses.replace(_spec(n, scheme), bc=((walls, walls), (0, 0), (0, 0)))
    Q = _state(spec)
    assert np.array_equal(_rhs(spec, Q, True), O.rhs(spec, Q))


@pytest.mark.parametrize("scheme", [W.WENO5JS, W.TENO5])
@pytest.mark.parametrize("n", SIZES)
def test_fast_smooth(n, scheme):
    spec = _spec(n, scheme)
    Q = W.random_smooth_state(spec, seed=43, amp=2e-3)
    dim = spec.dim
    alpha = O.wavespeeds(spec, Q)
    p = (spec.gamma - 1) * (Q[-1] - 0.5 * np.sum(Q[1:1 + dim] ** 2, axis=0) / Q[0])
    bound = sum(64 * np.finfo(np.float64).eps
                * (np.abs(Q[-1] + p).max() + alpha[a] * np.abs(Q).max()) / spec.h[a]
                for a in range(dim))
    assert np.abs(_rhs(spec, Q, False) - O.rhs(spec, Q)).max() <= bound


def test_stretched_rows():
    from paper_1905_00182_gb300 import ibfsa as ib
    lo, hi, x, m = W.stretched_axis(75, 0.04, 0.09, 41, 8, center=0.0)
    spec = dataclasses.replace(_spec((75, 6, 7), W.TENO5), lo=(lo, -1.0, -1.0), hi=(hi, 1.0, 1.0))
    Q = W.random_smooth_state(spec, seed=44, amp=2e-3, step=0.05)
    g = ib.Grid(spec, strict=True)
    g.set_mesh(0, x, m)
    g.set_state(Q)
    got = g.rhs().cpu().numpy()
    assert g.status() == 0
    g.close()
    assert np.array_equal(got, O.rhs(spec, Q, stretch=[(x, m), None, None]))
