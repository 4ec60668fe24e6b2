"""Characteristic-wise FP64 passes at the edges of their tiles (63 cells x 4 rows along x, 15 cells x 32 lines
along y and z), with a few blocks per multiprocessor and with many, against the oracle (arXiv:1905.00182,
Sec. 2): strict bit for bit; fast on smooth modes, per element within twice the bound of
test_gpu_conv_tiles.py (the projection to and from the fields adds as many roundings as the rest).
"""
import dataclasses

import numpy as np
import pytest

from oracle import oracle as O
from paper_1905_00182_gb300 import workloads as W
from tests.test_gpu_conv_tiles import _rhs, _spec, _state

pytestmark = pytest.mark.gpu

SIZES = [(33, 16), (64, 31), (97, 90), (32, 15, 16), (33, 16, 15), (65, 17, 31), (34, 17, 200)]


@pytest.mark.parametrize("scheme", [W.WENO5JS, W.TENO5])
@pytest.mark.parametrize("n", SIZES)
def test_strict_bits(n, scheme):
    spec = dataclasses.replace(_spec(n, scheme), charwise=True)
    Q = _state(spec)
    assert np.array_equal(_rhs(spec, Q, True), O.rhs(spec, Q, charwise=True))


@pytest.mark.parametrize("scheme", [W.WENO5JS, W.TENO5])
@pytest.mark.parametrize("n", SIZES)
def test_fast_smooth(n, scheme):
    spec = dataclasses.replace(_spec(n, scheme), charwise=True)
    Q = W.random_smooth_state(spec, seed=47, amp=2e-3)
    dim = spec.dim
    alpha = O.wavespeeds(spec, Q)
    p = (spec.gamma - 1) * (Q[-1] - 0.5 * np.sum(Q[1:1 + dim] ** 2, axis=0) / Q[0])
    bound = sum(128 * np.finfo(np.float64).eps
                * (np.abs(Q[-1] + p).max() + alpha[a] * np.abs(Q).max()) / spec.h[a]
                for a in range(dim))
    assert np.abs(_rhs(spec, Q, False) - O.rhs(spec, Q, charwise=True)).max() <= bound
