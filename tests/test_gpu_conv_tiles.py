"""FP64 convective passes at the edges of their tiles: lines in groups of 32, segments of up to
8 K - 1 cells with K = 1, 2 or 4 faces per thread chosen by the grid, against the oracle
(arXiv:1905.00182, Sec. 2).

Strict: bit for bit, on a state that mixes a quiescent region (exactly constant), rounding-level
noise, a smooth pulse and a contact step, so every path of TENO5 runs.  Fast: on smooth modes, per
element within 64 eps of the split-flux scale of each direction, summed over the directions.
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

SIZES = [(4, 9), (7, 8), (8, 7), (15, 33), (32, 16), (33, 31), (64, 65), (63, 127), (257, 130),
         (130, 401), (9, 8, 33), (33, 7, 16), (16, 34, 8), (65, 40, 34), (96, 70, 64)]


def _state(spec):
    Q = W.gaussian_pulse_state(spec, (0.3, 0.2, 0.1), amp=2e-2, halfwidth=0.15)
    X = W.mesh(spec)[0]
    Q = Q * np.where(X < -0.6, 1.05, 1.0)                 # contact step, constant beyond it
    rng = np.random.default_rng(3)
    noise = 1e-16 * rng.integers(-2, 3, size=Q.shape) * (X > 0.6)
    return Q + noise


def _rhs(spec, Q, strict):
    from paper_1905_00182_gb300 import ibfsa as ib
    g = ib.Grid(spec, strict=strict)
    g.set_state(Q)
    L = g.rhs().cpu().numpy()
    assert g.status() == 0
    g.close()
    return L


def _spec(n, scheme):
    dim = len(n)
    return W.GridSpec(dim=dim, n=tuple(n) + (1,) * (3 - dim), lo=(-1.0,) * 3, hi=(1.0,) * 3,
                      gamma=1.4, Re=0.0, qinf=W.freestream(dim, 1.4), scheme=scheme)


def _oracle(spec, Q):
    L = O.rhs(spec, Q)
    return L[0] if isinstance(L, tuple) else L


@pytest.mark.parametrize("scheme", [W.WENO5JS, W.TENO5])
@pytest.mark.parametrize("n", SIZES)
def test_strict_bits(n, scheme):
    spec = _spec(n, scheme)
    Q = _state(spec)
    assert np.array_equal(_rhs(spec, Q, True), _oracle(spec, Q))


@pytest.mark.parametrize("scheme", [W.WENO5JS, W.TENO5])
@pytest.mark.parametrize("n", SIZES)
def test_fast_smooth(n, scheme):
    spec = _spec(n, scheme)
    Q = W.random_smooth_state(spec, seed=41, amp=2e-3)
    dim = spec.dim
    alpha = O.wavespeeds(spec, Q)
    p = (spec.gamma - 1) * (Q[-1] - 0.5 * np.sum(Q[1:1 + dim] ** 2, axis=0) / Q[0])
    bound = sum(64 * np.finfo(np.float64).eps
                * (np.abs(Q[-1] + p).max() + alpha[a] * np.abs(Q).max()) / spec.h[a]
                for a in range(dim))
    assert np.abs(_rhs(spec, Q, False) - _oracle(spec, Q)).max() <= bound
